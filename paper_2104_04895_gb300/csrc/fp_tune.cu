// Autotuner of the rate kernel's tiles: times each candidate (branch chunk J dividing nb, q'-tile,
// threads per block) and the untuned default on a sample of q-points with the real kernel and remembers the fastest per
// (precision, one or several temperatures) in the context.  The sample is not the grid: a pair of the kernel over pairs
// whose partner lies outside has one value to write instead of two.  So the default stays unless a candidate beats it by
// more than 3 %.
#include <algorithm>
#include <cstring>
#include <vector>

#include "fp_internal.cuh"

namespace {
int tfail(fp_ctx* c, int code, const std::string& m) {
  c->err = m;
  return code;
}
}  // namespace

extern "C" int fp_autotune(fp_ctx* c, int nT, const double* T, double scalebroad, fp_rates_opts* opts,
                           double* best_ms) {
  if (!c || !opts) return FP_EINVAL;
  if (!c->have_modes) return tfail(c, FP_ESTATE, "fp_autotune: call fp_modes or fp_set_modes first");
  if (nT < 1 || nT > fp::kMaxT || !T) return tfail(c, FP_EINVAL, "fp_autotune: nT must be in [1, 8]");
  if (opts->precision < FP_PREC_FP64 || opts->precision > FP_PREC_DOUBLE_FLOAT)
    return tfail(c, FP_EINVAL, "fp_autotune: unknown precision");
  const int N = c->N, nb = c->nb;
  const int maxth = fp::max_tile_threads(c, *opts);
  // q sample: about 64 x 512^2 (q, q', q'') triples per trial (a few percent of a 512-point grid), and at
  // least 4 q-points, so that every candidate is timed on the same, bounded work
  long long want = (64LL * 512 * 512) / ((long long)N * N);
  int nq = (int)(want < 4 ? 4 : want);
  if (nq > N) nq = N;
  double* d_out = nullptr;
  if (cudaSetDevice(c->device) != cudaSuccess ||
      cudaMalloc(reinterpret_cast<void**>(&d_out), (size_t)nT * N * nb * sizeof(double)) != cudaSuccess)
    return tfail(c, FP_ENOMEM, "fp_autotune: cannot allocate the trial output");
  int* tt = c->tuned[opts->precision][nT == 1 ? 0 : 1];
  const int before[3] = {tt[0], tt[1], tt[2]};
  tt[0] = tt[1] = tt[2] = 0;  // the automatic tile of the trials is the untuned one
  double best = 1e300;
  int tile[3] = {0, 0, 0};
  auto trial = [&](int J, int t1, int th, double margin) {
    fp_rates_opts o = *opts;
    o.block_j0 = J;
    o.k1_tile = t1;
    o.threads = th;
    o.q_begin = 0;
    o.q_end = nq;
    o.no_graph = 1;
    o.mode_mask = nullptr;
    fp_stats st;
    double ms = 1e300;
    for (int rep = 0; rep < 3; ++rep) {  // the first run warms up
      if (fp_rates4_device(c, nT, T, scalebroad, &o, d_out, &st) != FP_OK) return false;  // a tile this device cannot hold
      if (rep) ms = std::min(ms, st.ms);
    }
    if (ms >= margin * best) return false;
    best = ms;
    for (int i = 0; i < 3; ++i) tile[i] = st.tile[i];
    return true;
  };
  trial(0, 0, 0, 1.0);
  const int base[3] = {tile[0], tile[1], tile[2]};
  bool tuned = false;
  const int t1s[] = {1, 2, 4};
  for (int J = 1; J <= nb; ++J) {
    if (nb % J || J * nb * nb > maxth) continue;
    const int th = (J * nb * nb + 31) / 32 * 32;  // extra threads would idle
    for (int t1 : t1s)
      if (J != base[0] || t1 != base[1] || th != base[2]) tuned = trial(J, t1, th, tuned ? 1.0 : 0.97) || tuned;
  }
  cudaFree(d_out);
  if (tile[0] == 0) {
    std::copy(before, before + 3, tt);
    return tfail(c, FP_EINVAL, "fp_autotune: no tile could run");
  }
  if (tuned) std::copy(tile, tile + 3, tt);
  opts->block_j0 = tile[0];
  opts->k1_tile = tile[1];
  opts->threads = tile[2];
  if (best_ms) *best_ms = best;
  c->err.clear();
  return FP_OK;
}

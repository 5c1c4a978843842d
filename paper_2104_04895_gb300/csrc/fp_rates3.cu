// Three-phonon RTA rates (paper Sec. 2.2, Eqs. tao0, 3phgamma, V3): fp_set_fc3 and fp_rates3.
//
// With k2 = q + k1 (mod G) and e(-k) = conj e(k) one vertex
//   W3(q, j; k1, j1; k2, j2) = sum_triplets sum_{abg} Phi3 / sqrt(M^3) e_a(q, j) e_b(k1, j1) conj(e_g(k2, j2))
//                              exp(i (k1.R_j - k2.R_k))
// is V+ of the partner q' = k1 and V- of the partner q' = -k1 (both with q'' = k2), so every (q, k1) pair
// serves both processes.  Time reversal gives the rates of -q (make_selection).
//
// One block owns a point q and a range of k1.  The phase is exp(-i q.R_k) exp(i k1.(R_j - R_k)), so the contraction with
// e(q) is done once per block, Psi[j][group][beta gamma] over the triplets of equal atoms (j, k) and D = R_j - R_k; per
// k1 the block forms A[j][(j b)(k g)] = sum_groups exp(i k1.D) Psi (nothing to do for D = 0), Y = A e(k1) and
// W = Y conj e(k2).  Thread o owns the entry (j, j1, j2).  The window is tested in FP32 with a proven margin and decided
// in FP64 in the operation order of the definition only inside it (as in fp_rates_kernel.cuh), and the accepted
// (entry, process) pairs of a warp are compacted and evaluated 32 at a time with 1/sigma and the Bose factors from
// tables per (j1, j2).  Sums run per entry, then over the entries of a j and over the k1 ranges in a fixed order.
//
// The FP64 pipe bounds this kernel.  Before, each (q, k1) took 1300 more FMAs for the assembly and e(q), an FP64 square
// root and 30 more operations for each of its 432 window tests, and every q ran: diamond 8^3 20.8 ms, now 4.2 ms.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <string>
#include <tuple>
#include <type_traits>
#include <vector>

#include "fp_pair_kernel.cuh"

namespace fp {
namespace {

struct Rates3Args {
  RatesArgs r;           // grid, modes, window and broadening fields (sigma_entry, sigma_entry_f32); qlist, mult
  int n3, G;
  const int* t3_meta;    // [n3][4] atom i and Rk, triplets by group
  const double* t3_fc;   // [n3][27] Phi3 / sqrt(Mi Mj Mk)
  const int* t3_start;   // [G + 1] triplets of a group (j, k, D = Rj - Rk)
  const int* g3_meta;    // [G][3] D
  const int* g3_start;   // [natoms^2 + 1] groups of (j, k), those with D = 0 first
  const double* bose;    // [nT][N nb] occupation numbers
  double2* psi;          // [nq_sel][nb][G][9]
  int psi_shared;        // the block keeps its Psi in shared memory
  int t0, nT_all;        // first temperature of this launch and their number in the call
  int nch, kchunk;       // k1 ranges per q
  double* partial;       // [nq_sel][nch][nb][nT_all]
  unsigned long long* counts;  // [2] accepted + and -, weighted by the selected modes a row stands for
};

__global__ void bose3_kernel(const double* omega, const double* T, int nT, long long nm, double* out) {
  const long long n = (long long)nT * nm;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double w = omega[i % nm];
    const double t = T[i / nm];
    out[i] = w > 0.0 ? 1.0 / expm1(kHbar * w / (kBoltzmann * t)) : 0.0;
  }
}

// Psi[qi][j][grp][beta gamma] = sum over the triplets of the group of exp(-i q.R_k) sum_alpha Phi3 e_alpha(q, j)
__global__ void psi3_kernel(Rates3Args p) {
  const RatesArgs& a = p.r;
  const long long n = (long long)a.nq_sel * a.nb * p.G * 9;
  for (long long o = blockIdx.x * (long long)blockDim.x + threadIdx.x; o < n; o += (long long)gridDim.x * blockDim.x) {
    const int bg = (int)(o % 9), grp = (int)((o / 9) % p.G), j = (int)((o / (9LL * p.G)) % a.nb);
    const int q = a.qlist[o / (9LL * p.G * a.nb)];
    const int g[3] = {q / (a.grid[1] * a.grid[2]), (q / a.grid[2]) % a.grid[1], q % a.grid[2]};
    const double2* e0 = a.evec + ((size_t)q * a.nb + j) * a.nb;
    Cx<double> sum = cmk<double>(0, 0);
    for (int Q = p.t3_start[grp]; Q < p.t3_start[grp + 1]; ++Q) {
      const int* m = p.t3_meta + 4 * Q;
      int e = 0;  // each term is below L, so e < 3 L
      for (int d = 0; d < 3; ++d) e += a.Lfac[d] * wrapi(-g[d] * m[1 + d], a.grid[d]);
      while (e >= a.L) e -= a.L;
      Cx<double> s = cmk<double>(0, 0);
      for (int al = 0; al < 3; ++al) {
        const double f = p.t3_fc[27 * (size_t)Q + al * 9 + bg];
        s.re = fma(f, e0[3 * m[0] + al].x, s.re);
        s.im = fma(f, e0[3 * m[0] + al].y, s.im);
      }
      cfma(sum, ld_tw<double>(a, e), s);
    }
    p.psi[o] = make_double2(sum.re, sum.im);
  }
}

__host__ __device__ constexpr int threads3(int nb) { return nb == 3 ? 32 : nb == 6 ? 224 : 256; }

// shared memory in bytes
struct Carve3 {
  size_t Psi, A, Y, E1, E2, Tw, Acc, W0, W1, W2, V1, V2, Iv8, F, B, Val, ExpT, Vf, PM, Hf, Ent, Mult, total;
};
__host__ __device__ inline Carve3 make_carve3(int nb, int G, int nT, bool psi) {
  Carve3 c;
  const size_t nb2 = (size_t)nb * nb, nb3 = nb2 * nb, nw = threads3(nb) / 32;
  size_t o = 0;
  auto put = [&](size_t bytes) {
    const size_t at = o;
    o += (bytes + 15) & ~size_t(15);
    return at;
  };
  c.Psi = put(psi ? (size_t)nb * G * 9 * 16 : 0);
  c.A = put(nb3 * 16);
  c.Y = put(nb3 * 16);
  c.E1 = put(nb2 * 16);
  c.E2 = put(nb2 * 16);
  c.Tw = put((size_t)G * 16);
  c.Acc = put(nb3 * nT * 8);
  c.W0 = put((size_t)nb * 8);
  c.W1 = put((size_t)nb * 8);
  c.W2 = put((size_t)nb * 8);
  c.V1 = put(3 * (size_t)nb * 8);
  c.V2 = put(3 * (size_t)nb * 8);
  c.Iv8 = put(2 * nb2 * 8);                 // 8/sigma or -1 (delta := 1), [process][j1][j2]
  c.F = put(2 * nb2 * 8);                   // (1/sigma) / (sqrt(pi) w' w'')
  c.B = put(2 * nb2 * nT * 8);              // Bose factors n' - n'' and (n' + n'' + 1) / 2
  c.Val = put(nw * 64 * 8);
  c.ExpT = put(kExpTab * 8);
  c.Vf = put(12 * (size_t)nb * 4);          // two-float velocities of k1 and k2
  c.PM = put(2 * nb2 * 8);                  // (P~, margin)
  c.Hf = put(3 * (size_t)nb * 4);           // FP32 frequencies of q, k1, k2
  c.Ent = put(nw * 64 * 2);
  c.Mult = put((size_t)nb);
  c.total = o;
  return c;
}

template <int NB>
__global__ void __launch_bounds__(threads3(NB), NB == 12 ? 1 : 2) rates3_kernel(Rates3Args p) {
  constexpr int NB2 = NB * NB, NB3 = NB2 * NB, NA = NB / 3, kThreads = threads3(NB);
  using C = Cx<double>;
  extern __shared__ __align__(16) unsigned char smem[];
  const RatesArgs& a = p.r;
  const int nT = a.nT, N = a.N, G = p.G;
  const Carve3 cv = make_carve3(NB, G, nT, p.psi_shared != 0);
  auto dbl = [&](size_t at) { return reinterpret_cast<double*>(smem + at); };
  auto flt = [&](size_t at) { return reinterpret_cast<float*>(smem + at); };
  C *sPsi = reinterpret_cast<C*>(smem + cv.Psi), *sA = reinterpret_cast<C*>(smem + cv.A), *sY = reinterpret_cast<C*>(smem + cv.Y);
  C *sE1 = reinterpret_cast<C*>(smem + cv.E1), *sE2 = reinterpret_cast<C*>(smem + cv.E2);
  C* sTw = reinterpret_cast<C*>(smem + cv.Tw);
  double *sAcc = dbl(cv.Acc), *sW0 = dbl(cv.W0), *sW1 = dbl(cv.W1), *sW2 = dbl(cv.W2), *sV1 = dbl(cv.V1), *sV2 = dbl(cv.V2);
  double *sIv8 = dbl(cv.Iv8), *sF = dbl(cv.F), *sB = dbl(cv.B), *sExpT = dbl(cv.ExpT);
  float *sVf = flt(cv.Vf), *sH0 = flt(cv.Hf), *sH1 = sH0 + NB, *sH2 = sH1 + NB;
  float2* sPM = reinterpret_cast<float2*>(smem + cv.PM);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double* sVal = dbl(cv.Val) + warp * 64;
  unsigned short* sEnt = reinterpret_cast<unsigned short*>(smem + cv.Ent) + warp * 64;
  unsigned char* sMult = smem + cv.Mult;
  const size_t NM = (size_t)N * NB;
  const int qi = blockIdx.x / p.nch, ch = blockIdx.x % p.nch;
  const int q = a.qlist[qi];
  const int g[3] = {q / (a.grid[1] * a.grid[2]), (q / a.grid[2]) % a.grid[1], q % a.grid[2]};
  const bool f32_sigma = a.dq_mode == 0;
  const double inv_sbdq = 1.0 / (a.sb * a.dq);
  const C* psi = reinterpret_cast<const C*>(p.psi) + (size_t)qi * NB * G * 9;
  if (p.psi_shared) {
    for (int o = tid; o < NB * G * 9; o += kThreads) sPsi[o] = psi[o];
    psi = sPsi;
  }
  for (int o = tid; o < NB; o += kThreads) {
    const double w = a.omega[(size_t)q * NB + o];
    sW0[o] = w;
    sH0[o] = __double2float_rn(w);
    sMult[o] = w > 0.0 ? a.mult[(size_t)q * NB + o] : 0;
  }
  for (int o = tid; o < kExpTab; o += kThreads) sExpT[o] = exp(-(double)o * kExpH);
  for (int o = tid; o < NB3 * nT; o += kThreads) sAcc[o] = 0.0;
  unsigned long long cplus = 0, cminus = 0;
  const int k_begin = ch * p.kchunk, k_end = min(N, k_begin + p.kchunk);
  for (int k1 = k_begin; k1 < k_end; ++k1) {
    const int g1[3] = {k1 / (a.grid[1] * a.grid[2]), (k1 / a.grid[2]) % a.grid[1], k1 % a.grid[2]};
    int g2[3];
    for (int d = 0; d < 3; ++d) {
      g2[d] = g[d] + g1[d];
      if (g2[d] >= a.grid[d]) g2[d] -= a.grid[d];
    }
    const int k2 = (g2[0] * a.grid[1] + g2[1]) * a.grid[2] + g2[2];
    __syncthreads();  // Psi; at later k1 the last one's terms
    for (int o = tid; o < NB2; o += kThreads) {
      sE1[o] = ld_e<double>(a, (size_t)k1 * NB2 + o);
      sE2[o] = ld_e<double>(a, (size_t)k2 * NB2 + o);
    }
    for (int o = tid; o < NB; o += kThreads) {
      sW1[o] = a.omega[(size_t)k1 * NB + o];
      sW2[o] = a.omega[(size_t)k2 * NB + o];
      sH1[o] = __double2float_rn(sW1[o]);
      sH2[o] = __double2float_rn(sW2[o]);
    }
    for (int o = tid; o < 3 * NB; o += kThreads) {
      const double v1 = a.vel[(size_t)k1 * NB * 3 + o], v2 = a.vel[(size_t)k2 * NB * 3 + o];
      sV1[o] = v1;
      sV2[o] = v2;
      const float h1 = __double2float_rn(v1), h2 = __double2float_rn(v2);
      sVf[o] = h1;
      sVf[3 * NB + o] = __double2float_rn(v1 - (double)h1);
      sVf[6 * NB + o] = h2;
      sVf[9 * NB + o] = __double2float_rn(v2 - (double)h2);
    }
    for (int o = tid; o < G; o += kThreads) {
      const int* D = p.g3_meta + 3 * o;
      int e = 0;
      for (int d = 0; d < 3; ++d) e += a.Lfac[d] * wrapi(g1[d] * D[d], a.grid[d]);
      while (e >= a.L) e -= a.L;
      sTw[o] = ld_tw<double>(a, e);
    }
    __syncthreads();
    for (int o = tid; o < NB3; o += kThreads) {
      const int j = o / NB2, b = (o / NB) % NB, c = o % NB, jk = b / 3 * NA + c / 3, bg = (b % 3) * 3 + c % 3;
      C s = cmk<double>(0, 0);
      int gi = p.g3_start[jk];
      const int g_end = p.g3_start[jk + 1];
      if (gi < g_end && p.g3_meta[3 * gi] == 0 && p.g3_meta[3 * gi + 1] == 0 && p.g3_meta[3 * gi + 2] == 0) {
        s = psi[(j * G + gi) * 9 + bg];
        ++gi;
      }
      for (; gi < g_end; ++gi) cfma(s, sTw[gi], psi[(j * G + gi) * 9 + bg]);
      sA[o] = s;
    }
    // tables per (process, j1, j2): + v(k1) - v(k2), - -v(k1) - v(k2)
    for (int o = kThreads - 1 - tid; o < 2 * NB2; o += kThreads) {
      const int pr = o / NB2, j1 = (o / NB) % NB, j2 = o % NB;
      double iv = -1.0;
      if (f32_sigma) {
        float inv;
        sigma_entry_f32(a, sVf + 3 * j1, sVf + 3 * NB + 3 * j1, pr ? -1.f : 1.f, sVf + 6 * NB + 3 * j2,
                        sVf + 9 * NB + 3 * j2, sV1 + 3 * j1, sV2 + 3 * j2, sPM + o, &inv);
        if (inv >= 0.f) {
          const double sg = pr ? -1.0 : 1.0;
          const double dx = sg * sV1[3 * j1] - sV2[3 * j2], dy = sg * sV1[3 * j1 + 1] - sV2[3 * j2 + 1],
                       dz = sg * sV1[3 * j1 + 2] - sV2[3 * j2 + 2];
          iv = rsqrt(fma(dx, dx, fma(dy, dy, dz * dz))) * inv_sbdq;
        }
      } else {
        double ex[2];
        float inv;
        sigma_entry(a, sV1 + 3 * j1, pr ? -1.0 : 1.0, sV2 + 3 * j2, ex);
        sigma_f_from_exact(ex, sPM + o, &inv);
        iv = ex[1];
      }
      sIv8[o] = iv >= 0.0 ? 8.0 * iv : -1.0;
      sF[o] = (iv >= 0.0 ? iv * kInvSqrtPi : 1.0) / (sW1[j1] * sW2[j2]);  // not used at zero frequency
    }
    for (int o = tid; o < 2 * NB2 * nT; o += kThreads) {
      const int t = o / (2 * NB2), pr = (o / NB2) % 2, j1 = (o / NB) % NB, j2 = o % NB;
      const double *n = p.bose + (size_t)(p.t0 + t) * NM, n1 = n[(size_t)k1 * NB + j1], n2 = n[(size_t)k2 * NB + j2];
      sB[o] = pr == 0 ? n1 - n2 : 0.5 * (n1 + n2 + 1.0);
    }
    __syncthreads();
    for (int o = tid; o < NB3; o += kThreads) {
      const int j = o / NB2, j1 = (o / NB) % NB, c = o % NB;
      C s = cmk<double>(0, 0);
#pragma unroll
      for (int b = 0; b < NB; ++b) cfma(s, sE1[j1 * NB + b], sA[(j * NB + b) * NB + c]);
      sY[o] = s;
    }
    __syncthreads();
    for (int o0 = warp * 32; o0 < NB3; o0 += kThreads) {
      const int o = o0 + lane;
      const int j = o / NB2, j1 = (o / NB) % NB, j2 = o % NB;
      // accepted processes of this entry: bit 0 (+), bit 1 (-)
      unsigned acc = 0;
      const unsigned mult = o < NB3 ? sMult[j] : 0u;
      if (mult && sH1[j1] != 0.f && sH2[j2] != 0.f) {
        const float h = sH0[j], h1 = sH1[j1], h2 = sH2[j2], sS = kRelS * ((h + h1) + h2);
#pragma unroll
        for (int pr = 0; pr < 2; ++pr) {
          const float2 pm = sPM[pr * NB2 + j1 * NB + j2];
          const float d = fabsf((pr ? h - h1 : h + h1) - h2), M = sS + pm.y;
          if (d < pm.x - M) {
            acc |= 1u << pr;
          } else if (d <= pm.x + M) {  // inside the rounding of the prefilter: decided in FP64
            double ex[2];
            sigma_entry(a, sV1 + 3 * j1, pr ? -1.0 : 1.0, sV2 + 3 * j2, ex);
            const double w = sW0[j], w1 = sW1[j1];
            if (fabs(__dsub_rn(pr ? __dsub_rn(w, w1) : __dadd_rn(w, w1), sW2[j2])) <= ex[0]) acc |= 1u << pr;
          }
        }
      }
      cplus += (acc & 1u) * mult;
      cminus += (acc >> 1) * mult;
      const unsigned b0 = __ballot_sync(0xffffffffu, acc & 1u), b1 = __ballot_sync(0xffffffffu, acc & 2u);
      const unsigned below = (1u << lane) - 1u;
      const int n0 = __popc(b0), total = n0 + __popc(b1);
      const int p0 = __popc(b0 & below), p1 = n0 + __popc(b1 & below);
      if (acc & 1u) sEnt[p0] = (unsigned short)lane;
      if (acc & 2u) sEnt[p1] = (unsigned short)(lane | 32);
      __syncwarp();
      for (int i = lane; i < total; i += 32) {
        const unsigned en = sEnt[i];
        const int oe = o0 + (int)(en & 31u), pr = (int)(en >> 5);
        const int ej = oe / NB2, e1 = (oe / NB) % NB, e2 = oe % NB, e = pr * NB2 + e1 * NB + e2;
        C W = cmk<double>(0, 0);
#pragma unroll
        for (int c = 0; c < NB; ++c) cfma_conj(W, sY[(ej * NB + e1) * NB + c], sE2[e2 * NB + c]);
        const double w = sW0[ej], w1 = sW1[e1];
        const double dw = __dsub_rn(pr ? __dsub_rn(w, w1) : __dadd_rn(w, w1), sW2[e2]);
        double v = (W.re * W.re + W.im * W.im) * sF[e];
        const double iv8 = sIv8[e];
        if (__double2hiint(iv8) >= 0) v *= pair_exp_neg64(dw * iv8, sExpT);
        sVal[i] = v;
      }
      __syncwarp();
      if (acc) {
        const double v0 = (acc & 1u) ? sVal[p0] : 0.0, v1 = (acc & 2u) ? sVal[p1] : 0.0;
        for (int t = 0; t < nT; ++t) {
          const double* B = sB + 2 * t * NB2 + j1 * NB + j2;
          sAcc[(size_t)o * nT + t] = fma(v0, B[0], fma(v1, B[NB2], sAcc[(size_t)o * nT + t]));
        }
      }
      __syncwarp();
    }
  }
  __syncthreads();
  for (int o = tid; o < NB * nT; o += kThreads) {
    const int j = o / nT, t = o % nT;
    double s = 0.0;
    for (int e = j * NB2; e < (j + 1) * NB2; ++e) s += sAcc[(size_t)e * nT + t];
    p.partial[((size_t)blockIdx.x * NB + j) * p.nT_all + p.t0 + t] = s;
  }
  for (int off = 16; off > 0; off >>= 1) {
    cplus += __shfl_down_sync(0xffffffffu, cplus, off);
    cminus += __shfl_down_sync(0xffffffffu, cminus, off);
  }
  if (lane == 0 && p.t0 == 0) {
    if (cplus) atomicAdd(p.counts, cplus);
    if (cminus) atomicAdd(p.counts + 1, cminus);
  }
}

// rates[t][q][j] = pref / w sum_ranges partial, in order, for the selected modes; the others stay zero
__global__ void reduce3_kernel(Rates3Args p, double pref, double* rates) {
  const RatesArgs& a = p.r;
  const long long n = (long long)p.nT_all * a.q_out_n * a.nb;
  const long long o = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (o >= n) return;
  const int j = (int)(o % a.nb);
  const int q = a.q_out_begin + (int)((o / a.nb) % a.q_out_n);
  const int t = (int)(o / ((long long)a.nb * a.q_out_n));
  const double w = a.omega[(size_t)q * a.nb + j];
  if (!a.sel[(size_t)q * a.nb + j] || !(w > 0.0)) return;
  const double* s = p.partial + (((size_t)a.qpos[q] * p.nch) * a.nb + j) * p.nT_all + t;
  double sum = 0.0;
  for (int ch = 0; ch < p.nch; ++ch) sum += s[(size_t)ch * a.nb * p.nT_all];
  rates[((size_t)t * a.N + q) * a.nb + j] = pref * sum / w;
}

const void* rates3_ptr(int nb) {
  switch (nb) {
    case 3: return reinterpret_cast<const void*>(&rates3_kernel<3>);
    case 6: return reinterpret_cast<const void*>(&rates3_kernel<6>);
    case 12: return reinterpret_cast<const void*>(&rates3_kernel<12>);
    default: return nullptr;
  }
}

int fail3(fp_ctx* c, int code, const std::string& msg) {
  c->err = msg;
  return code;
}

}  // namespace
}  // namespace fp

using namespace fp;

#define R3_CUDA(call)                                                                              \
  do {                                                                                             \
    cudaError_t e_ = (call);                                                                       \
    if (e_ != cudaSuccess)                                                                         \
      return fail3(c, e_ == cudaErrorMemoryAllocation ? FP_ENOMEM : FP_ECUDA,                      \
                   std::string(#call) + ": " + cudaGetErrorString(e_));                            \
  } while (0)

extern "C" int fp_set_fc3(fp_ctx* c, int n_fc3, const fp_fc3* fc3) {
  if (!c) return FP_EINVAL;
  if (n_fc3 < 0 || (n_fc3 > 0 && !fc3)) return fail3(c, FP_EINVAL, "fp_set_fc3: bad triplet list");
  const int na = c->natoms;
  // triplets by group (j, k, D = Rj - Rk), groups by (j, k) with D = 0 first; Phi3 / sqrt(Mi Mj Mk)
  std::map<std::tuple<int, int, int, int, int>, std::vector<int>> groups;
  for (int b = 0; b < n_fc3; ++b) {
    const fp_fc3& f = fc3[b];
    if (f.i < 0 || f.j < 0 || f.k < 0 || f.i >= na || f.j >= na || f.k >= na)
      return fail3(c, FP_EINVAL, "fp_set_fc3: atom index out of range");
    const int D[3] = {f.Rj[0] - f.Rk[0], f.Rj[1] - f.Rk[1], f.Rj[2] - f.Rk[2]};
    groups[std::make_tuple(f.j * na + f.k, D[0] || D[1] || D[2] ? 1 : 0, D[0], D[1], D[2])].push_back(b);
  }
  std::vector<int> start(1, 0), tmeta, meta, gstart(na * na + 1, 0);
  std::vector<double> val;
  for (const auto& kv : groups) {
    gstart[std::get<0>(kv.first) + 1]++;
    meta.push_back(std::get<2>(kv.first));
    meta.push_back(std::get<3>(kv.first));
    meta.push_back(std::get<4>(kv.first));
    for (int b : kv.second) {
      const fp_fc3& f = fc3[b];
      tmeta.push_back(f.i);
      for (int d = 0; d < 3; ++d) tmeta.push_back(f.Rk[d]);
      const double m = std::sqrt(c->mass[f.i] * c->mass[f.j] * c->mass[f.k]);
      for (int x = 0; x < 27; ++x) val.push_back(f.fc[x] / m);
    }
    start.push_back((int)tmeta.size() / 4);
  }
  for (int k = 0; k < na * na; ++k) gstart[k + 1] += gstart[k];
  R3_CUDA(cudaSetDevice(c->device));
  c->have_fc3 = false;
  auto put = [&](auto*& dst, const auto& src) -> cudaError_t {
    using T = typename std::remove_reference<decltype(*dst)>::type;
    if (dst) cudaFree(dst);
    dst = nullptr;
    cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&dst), std::max<size_t>(1, src.size()) * sizeof(T));
    if (e != cudaSuccess) return e;
    return cudaMemcpy(dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice);
  };
  R3_CUDA(put(c->d_t3_start, start));
  R3_CUDA(put(c->d_t3_meta, tmeta));
  R3_CUDA(put(c->d_t3_fc, val));
  R3_CUDA(put(c->d_g3_meta, meta));
  R3_CUDA(put(c->d_g3_start, gstart));
  c->G3 = (int)groups.size();
  c->n3 = n_fc3;
  c->have_fc3 = true;
  return FP_OK;
}

extern "C" int fp_rates3(fp_ctx* c, int nT, const double* T, double scalebroad, const fp_rates_opts* opts,
                         double* rates, fp_stats* stats) {
  if (!c) return FP_EINVAL;
  if (!rates) return fail3(c, FP_EINVAL, "fp_rates3: NULL output");
  if (!c->have_fc3) return fail3(c, FP_ESTATE, "fp_rates3: call fp_set_fc3 first");
  if (!c->have_modes) return fail3(c, FP_ESTATE, "fp_rates3: call fp_modes or fp_set_modes first");
  if (nT < 1 || nT > fp::kMaxT || !T) return fail3(c, FP_EINVAL, "fp_rates3: nT must be in [1, 8]");
  for (int i = 0; i < nT; ++i)
    if (!(T[i] > 0.0) || !std::isfinite(T[i])) return fail3(c, FP_EINVAL, "fp_rates3: temperatures must be > 0");
  if (!(scalebroad > 0.0) || !std::isfinite(scalebroad)) return fail3(c, FP_EINVAL, "fp_rates3: scalebroad must be > 0");
  fp_rates_opts o;
  fp_default_opts(&o);
  if (opts) o = *opts;
  if (o.window == 0.0) o.window = 2.0;
  if (o.sigma_min == 0.0) o.sigma_min = 1e-10;
  if (!(o.window > 0.0) || !(o.sigma_min > 0.0)) return fail3(c, FP_EINVAL, "fp_rates3: window, sigma_min > 0");
  if (o.dq_mode != 0 && o.dq_mode != 1) return fail3(c, FP_EINVAL, "fp_rates3: dq_mode must be 0 or 1");
  const int N = c->N, nb = c->nb;
  const int q_end = o.q_end > 0 ? o.q_end : N;
  if (o.q_begin < 0 || o.q_begin > q_end || q_end > N) return fail3(c, FP_EINVAL, "fp_rates3: bad q range");
  const void* k = rates3_ptr(nb);
  if (!k) return fail3(c, FP_EINVAL, "fp_rates3: nb must be 3, 6 or 12");
  const size_t nm = (size_t)N * nb;
  // Psi in shared memory while two blocks fit an SM (one with twelve branches), else read from the table; temperatures
  // in as many launches as their sums per entry need
  const size_t most = 227 * 1024;
  int nTb = nT;
  while (nTb > 1 && make_carve3(nb, c->G3, nTb, false).total > most) --nTb;
  const bool psi_shared = make_carve3(nb, c->G3, nTb, true).total <= (nb == 12 ? most : most / 2);
  const size_t smem = make_carve3(nb, c->G3, nTb, psi_shared).total;
  if (smem > most) return fail3(c, FP_EINVAL, "fp_rates3: tables do not fit in shared memory");
  R3_CUDA(cudaSetDevice(c->device));
  cudaStream_t s = c->stream;
  // one point of each pair {q, -q}; the other options of `o` do not apply
  fp_rates_opts so;
  fp_default_opts(&so);
  so.mode_mask = o.mode_mask;
  so.q_begin = o.q_begin;
  so.q_end = o.q_end;
  Selection sel;
  std::string err;
  int rc = make_selection(c, so, true, &sel, &err);
  if (rc) return fail3(c, rc, "fp_rates3: " + err);
  const int nq = (int)sel.qlist.size();
  // k1 ranges: enough blocks to fill the SMs about eight times over, so that the last wave costs little, of 16 points or
  // more, and of 4 where those would leave half of the resident blocks empty (measured, 16 against 4: diamond 2x2x2 67 ->
  // 49 us, 3x3x3 142 -> 64, 4x4x4 157 -> 137, LiCoO2 3x3x3 927 -> 300; but simple cubic 6x6x6 216 -> 277, LiCoO2 5x4x3
  // 1053 -> 1085)
  int nsm = 0;
  R3_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, c->device));
  int nch = nq > 0 ? (nsm * 16 + nq - 1) / nq : 1;
  const int least = 2LL * nq * ((N + 15) / 16) < (long long)nsm * (nb == 12 ? 1 : 2) ? 4 : 16;
  nch = std::max(1, std::min(nch, (N + least - 1) / least));
  const int kchunk = (N + nch - 1) / nch;
  nch = (N + kchunk - 1) / kchunk;
  // working memory, kept in the context: T, occupation table, counts, partial sums, rates, selection, Psi
  const size_t part = std::max<size_t>(1, (size_t)nq * nch * nb * nT);
  const size_t sizes[] = {nT * sizeof(double), nT * nm * sizeof(double), 2 * sizeof(unsigned long long), part * sizeof(double),
                          nT * nm * sizeof(double), nm, nm, (size_t)N * sizeof(int), (size_t)N * sizeof(int),
                          std::max<size_t>(1, (size_t)nq * nb * c->G3 * 9) * sizeof(double2)};
  size_t off[11] = {0};
  for (int i = 0; i < 10; ++i) off[i + 1] = off[i] + ((sizes[i] + 255) & ~size_t(255));
  if (c->scratch_cap < off[10]) {
    if (c->d_scratch) cudaFree(c->d_scratch);
    c->d_scratch = nullptr;
    c->scratch_cap = 0;
    R3_CUDA(cudaMalloc(reinterpret_cast<void**>(&c->d_scratch), off[10]));
    c->scratch_cap = off[10];
  }
  unsigned char* base = c->d_scratch;
  double *dT = reinterpret_cast<double*>(base), *dn = reinterpret_cast<double*>(base + off[1]);
  unsigned long long* dc = reinterpret_cast<unsigned long long*>(base + off[2]);
  double* dr = reinterpret_cast<double*>(base + off[4]);
  Rates3Args a;
  std::memset(&a, 0, sizeof(a));
  RatesArgs& r = a.r;
  r.N = N;
  r.nb = nb;
  r.natoms = c->natoms;
  r.nT = nT;
  r.L = c->L;
  for (int d = 0; d < 3; ++d) {
    r.grid[d] = c->grid[d];
    r.Lfac[d] = c->L / c->grid[d];
  }
  r.omega = c->d_omega;
  r.evec = c->d_evec;
  r.vel = c->d_vel;
  r.tw = c->d_tw;
  r.sb = scalebroad;
  r.window = o.window;
  r.sigma_min = o.sigma_min;
  const double* B = c->rec;
  const double detB = B[0] * (B[4] * B[8] - B[5] * B[7]) - B[1] * (B[3] * B[8] - B[5] * B[6]) +
                      B[2] * (B[3] * B[7] - B[4] * B[6]);
  r.dq = std::cbrt(std::fabs(detB) / (double)N);
  r.dq_mode = o.dq_mode;
  for (int i = 0; i < 9; ++i) r.rec[i] = B[i];
  r.mult = base + off[5];
  r.sel = base + off[6];
  r.qlist = reinterpret_cast<int*>(base + off[7]);
  r.qpos = reinterpret_cast<int*>(base + off[8]);
  r.q_out_begin = sel.q_out_begin;
  r.q_out_n = sel.q_out_end - sel.q_out_begin;
  r.nq_sel = nq;
  a.n3 = c->n3;
  a.G = c->G3;
  a.t3_start = c->d_t3_start;
  a.t3_meta = c->d_t3_meta;
  a.t3_fc = c->d_t3_fc;
  a.psi = reinterpret_cast<double2*>(base + off[9]);
  a.psi_shared = psi_shared ? 1 : 0;
  a.nT_all = nT;
  a.g3_meta = c->d_g3_meta;
  a.g3_start = c->d_g3_start;
  a.bose = dn;
  a.nch = nch;
  a.kchunk = kchunk;
  a.partial = reinterpret_cast<double*>(base + off[3]);
  a.counts = dc;
  const double pref = kPi * kHbar * kConv * kConv * kConv / (4.0 * (double)N);
  R3_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  R3_CUDA(cudaMemcpyAsync(dT, T, nT * sizeof(double), cudaMemcpyHostToDevice, s));
  R3_CUDA(cudaMemcpyAsync(base + off[5], sel.mult.data(), nm, cudaMemcpyHostToDevice, s));
  R3_CUDA(cudaMemcpyAsync(base + off[6], sel.sel.data(), nm, cudaMemcpyHostToDevice, s));
  if (nq > 0) R3_CUDA(cudaMemcpyAsync(base + off[7], sel.qlist.data(), nq * sizeof(int), cudaMemcpyHostToDevice, s));
  R3_CUDA(cudaMemcpyAsync(base + off[8], sel.qpos.data(), (size_t)N * sizeof(int), cudaMemcpyHostToDevice, s));
  R3_CUDA(cudaMemsetAsync(dr, 0, nT * nm * sizeof(double), s));
  R3_CUDA(cudaMemsetAsync(dc, 0, 2 * sizeof(unsigned long long), s));
  R3_CUDA(cudaEventRecord(c->ev0, s));
  bose3_kernel<<<256, 256, 0, s>>>(c->d_omega, dT, nT, (long long)nm, dn);
  R3_CUDA(cudaGetLastError());
  if (nq > 0) {
    psi3_kernel<<<4 * nsm, 256, 0, s>>>(a);
    R3_CUDA(cudaGetLastError());
    for (int t0 = 0; t0 < nT; t0 += nTb) {
      a.t0 = t0;
      r.nT = std::min(nTb, nT - t0);
      void* args[] = {&a};
      R3_CUDA(cudaLaunchKernel(k, dim3(nq * nch), dim3(threads3(nb)), args, smem, s));
    }
    const long long n = (long long)nT * r.q_out_n * nb;
    reduce3_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a, pref, dr);
    R3_CUDA(cudaGetLastError());
  }
  R3_CUDA(cudaEventRecord(c->ev1, s));
  unsigned long long cnt[2] = {0, 0};
  R3_CUDA(cudaMemcpyAsync(rates, dr, nT * nm * sizeof(double), cudaMemcpyDeviceToHost, s));
  R3_CUDA(cudaMemcpyAsync(cnt, dc, sizeof(cnt), cudaMemcpyDeviceToHost, s));
  R3_CUDA(cudaStreamSynchronize(s));
  trim_scratch(c);
  if (stats) {
    std::memset(stats, 0, sizeof(*stats));
    double nsel = 0;
    for (int qq = o.q_begin; qq < q_end; ++qq)
      for (int j = 0; j < nb; ++j) nsel += (!o.mode_mask || o.mode_mask[(size_t)qq * nb + j]) ? 1 : 0;
    stats->candidates = 2.0 * nsel * (double)N * nb * nb;
    stats->accepted[0] = (double)cnt[0];
    stats->accepted[1] = (double)cnt[1];
    // per evaluated (q, k1): the assembly over the groups (9 nb G) and two nb^4 contractions
    stats->flops = (double)nq * N * 8.0 * (9.0 * nb * c->G3 + 2.0 * nb * nb * nb * nb);
    float ms = 0.f;
    cudaEventElapsedTime(&ms, c->ev0, c->ev1);
    stats->ms = ms;
    stats->tile[2] = threads3(nb);
    stats->tile[3] = nq * nch;
  }
  return FP_OK;
}

namespace fp {
namespace {

// RTA thermal conductivity (the tensor the paper's rates feed, Sec. 2.1): kappa_ab(T) = k_B / (N V)
// sum_l c(x_l) v_a v_b / rate_l, c(x) = x^2 e^x / (e^x - 1)^2 = (x/2 / sinh(x/2))^2, x = hbar w / (k_B T).
// One CTA per temperature; per-thread sums over a fixed mode stride, then a fixed-order tree in shared memory.
__global__ void kappa_kernel(const double* omega, const double* vel, const double* rates, const double* T, int nm,
                             double scale, double* kappa) {
  __shared__ double s[9][256];
  const int t = blockIdx.x, tid = threadIdx.x;
  double acc[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
  for (int m = tid; m < nm; m += blockDim.x) {
    const double w = omega[m], r = rates[(size_t)t * nm + m];
    if (!(w > 0.0) || !(r > 0.0)) continue;
    const double h = 0.5 * fp::kHbar * w / (fp::kBoltzmann * T[t]);
    const double ch = h / sinh(h);
    const double f = ch * ch / r;
    const double* v = vel + 3 * (size_t)m;
    for (int a = 0; a < 3; ++a)
      for (int b = 0; b < 3; ++b) acc[3 * a + b] += f * v[a] * v[b];
  }
  for (int k = 0; k < 9; ++k) s[k][tid] = acc[k];
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (tid < w)
      for (int k = 0; k < 9; ++k) s[k][tid] += s[k][tid + w];
    __syncthreads();
  }
  if (tid < 9) kappa[9 * t + tid] = scale * s[tid][0];
}

}  // namespace
}  // namespace fp

extern "C" int fp_kappa_rta(fp_ctx* c, int nT, const double* T, const double* rates, double* kappa) {
  if (!c) return FP_EINVAL;
  if (!T || !rates || !kappa || nT < 1 || nT > fp::kMaxT) return fail3(c, FP_EINVAL, "fp_kappa_rta: bad arguments");
  for (int i = 0; i < nT; ++i)
    if (!(T[i] > 0.0) || !std::isfinite(T[i])) return fail3(c, FP_EINVAL, "fp_kappa_rta: temperatures must be > 0");
  if (!c->have_modes) return fail3(c, FP_ESTATE, "fp_kappa_rta: call fp_modes or fp_set_modes first");
  const int nm = c->N * c->nb;
  const double* A = c->lattice;
  const double vol = std::fabs(A[0] * (A[4] * A[8] - A[5] * A[7]) - A[1] * (A[3] * A[8] - A[5] * A[6]) +
                               A[2] * (A[3] * A[7] - A[4] * A[6]));
  // k_B [J/K] (A/ps)^2 ps / A^3 = 1.380649e-23 * 1e4 * 1e-12 / 1e-30 W/(m K)
  const double scale = 1.380649e-23 * 1e4 * 1e-12 / 1e-30 / ((double)c->N * vol);
  R3_CUDA(cudaSetDevice(c->device));
  cudaStream_t s = c->stream;
  double *dT = nullptr, *dr = nullptr, *dk = nullptr;
  auto cleanup = [&]() {
    cudaFree(dT);
    cudaFree(dr);
    cudaFree(dk);
  };
  bool ok = cudaMalloc(&dT, nT * sizeof(double)) == cudaSuccess &&
            cudaMalloc(&dr, (size_t)nT * nm * sizeof(double)) == cudaSuccess &&
            cudaMalloc(&dk, 9 * nT * sizeof(double)) == cudaSuccess &&
            cudaMemcpyAsync(dT, T, nT * sizeof(double), cudaMemcpyHostToDevice, s) == cudaSuccess &&
            cudaMemcpyAsync(dr, rates, (size_t)nT * nm * sizeof(double), cudaMemcpyHostToDevice, s) == cudaSuccess;
  if (ok) {
    kappa_kernel<<<nT, 256, 0, s>>>(c->d_omega, c->d_vel, dr, dT, nm, scale, dk);
    ok = cudaGetLastError() == cudaSuccess &&
         cudaMemcpyAsync(kappa, dk, 9 * nT * sizeof(double), cudaMemcpyDeviceToHost, s) == cudaSuccess &&
         cudaStreamSynchronize(s) == cudaSuccess;
  }
  cleanup();
  if (!ok) return fail3(c, FP_ECUDA, "fp_kappa_rta: CUDA call failed");
  return FP_OK;
}

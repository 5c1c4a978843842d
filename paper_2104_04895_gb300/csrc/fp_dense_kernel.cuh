// Mixed-precision four-phonon rate kernel: the sums of fp_rates_kernel.cuh (ordered q', k1 <= k2, six candidates per
// entry, the FP32 form) with every FP32 vertex and weight product formed by the same operations in the same order.  Only dw
// (one sum of tabulated pairs instead of a chain of three, the last bits of the float that enters the Gaussian) and the
// order of the compensated sums differ: rates move by at most 2e-12, 1e-13 in the 2-norm (six crystals and grids up to
// 8x8x8, one and eight temperatures).
//
// The path is bound by instruction issue; this layout spends fewer instructions per entry (j0, x, y, j3):
//   - the tables of a grid point that the loop over k2 needs lie in one record (record_kernel): one 16-byte load per
//     thread and k2, held in registers while the last k2 is worked on, two barriers per k2 instead of three;
//   - thread (j0, x, s) builds the A row of component s and, after a barrier, owns branch s of k3: its column of
//     T = A conj(e3) stays in registers and W of every y follows from broadcast reads of e2, without a T block in shared
//     memory; its sigma entries of v(k1, x) are constants of a k2;
//   - the two +- candidates, nearly all accepted terms, are evaluated for every entry with the window as a select and dw
//     as one two-float sum of tabulated pairs (w0 + wx) - (wy + w3) and (w0 - wx) + (wy - w3); the other four, which
//     single lanes accept now and then, are compacted per warp and evaluated 32 at a time;
//   - window bounds (P - margin, P + margin) come from the tables, with the margin for the largest frequencies of the
//     block: candidates between the two are decided in FP64 as before.
// The loop over y is unrolled fully with one temperature (37.9 ms on diamond 6x6x6; by twos 39.7) and by twos with
// several (diamond 6x6x6, 8 temperatures: 68.6 ms; fully 82.2).
// Measured (GB300, ordered float kernel -> this one): diamond 8x8x8 760 -> 473 ms, 6x6x6 with 8 temperatures 114.0 ->
// 68.6 ms, BAs 7x6x6 94.4 -> 78.0 ms, simple cubic 7x6x6 9.69 -> 5.1 ms.  On diamond 5x5x5 the schedulers issue in 61 %
// of the cycles (14 warps per SM; 58 % of the instructions are on the FMA pipes) and the FP64 pipe is 1 % busy.
#pragma once
#include "fp_rates_kernel.cuh"

namespace fp {
namespace {

constexpr int kDenseGroup = 6;   // y values compacted at once (four rare candidates each: 24 bits of a lane's mask)
constexpr int kDenseCap = 128;   // list entries per warp and round

// Blocks per SM of the register budget.  Six branches: two (37.9 ms on diamond 6x6x6; three spill and take 48.6).  Three
// branches, whose blocks are one warp: four times their largest size (5.1 ms on simple cubic 7x6x6; three 5.8, six 8.3).
__host__ __device__ constexpr int dense_blocks_for(int nb) { return nb == 3 ? 4 : 2; }

// record of a grid point, in floats: e (2 nb^2), group phases (2 G), omega as two floats (nb, nb), velocity as two
// floats (3 nb, 3 nb), weights ((1+n)/w, n/w) (nT nb pairs)
struct DenseRecord {
  int E, Tw, H, L, VH, VL, W, size;
};
__host__ __device__ inline DenseRecord make_record(int nb, int G, int nT) {
  DenseRecord r;
  int o = 0;
  r.E = o; o += 2 * nb * nb;
  r.Tw = o; o += 2 * G;
  r.W = o; o += 2 * nT * nb;
  r.H = o; o += nb;
  r.L = o; o += nb;
  r.VH = o; o += 3 * nb;
  r.VL = o; o += 3 * nb;
  r.size = (o + 3) & ~3;
  return r;
}

// shared memory in bytes
struct DenseCarve {
  size_t Rec, E0, E1, Psi, TwQ, A, X, T1, T0, T3, T2, U, F0, F1, H0, H1, VH1, VL1, W2, Val, Ent, KLs, KLg, Mult, total;
};
__host__ __device__ inline DenseCarve make_dense_carve(int nb, int J, int G, int nquart, int nT, int threads) {
  DenseCarve c;
  const size_t nb2 = (size_t)nb * nb, na = nb / 3, nw = ((size_t)threads + 31) / 32;
  size_t o = 0;
  auto put = [&](size_t bytes) {
    const size_t at = o;
    o += (bytes + 15) & ~size_t(15);
    return at;
  };
  auto max2 = [](size_t a, size_t b) { return a > b ? a : b; };
  c.Rec = put((size_t)make_record(nb, G, nT).size * 4 * 4);  // two buffers of the records of k2 and k3
  c.E0 = put((size_t)J * nb * 8);
  c.E1 = put(nb2 * 8);
  c.Psi = put((size_t)J * nb * G * 9 * 8);
  c.TwQ = put((size_t)nquart * 8);
  // (j0, x) blocks padded by 16 bytes; the products e0 e1 in the prologue, the row sums at the end
  c.A = put(max2((size_t)J * nb * (nb2 + 2) * 8, (size_t)threads * 8 * nT));
  c.X = put((size_t)J * nb * 16);   // w0 + wx and w0 - wx as two floats
  c.T1 = put(nb2 * 16);             // -v2 - v3, [y][j3]: (P - M, P + M, 1/sigma, P + M of v2 - v3)
  c.T0 = put(nb2 * 8);              // v2 - v3: (P - M, 1/sigma)
  c.T3 = put(nb2 * 16);             // -v1 - v3, [x][j3], likewise with v1
  c.T2 = put(nb2 * 8);
  c.U = put(nb2 * 16);              // wy + w3 and wy - w3 as two floats, NaN where a frequency is zero
  c.F0 = put((size_t)nT * J * 4);
  c.F1 = put((size_t)nT * nb * 8);
  c.H0 = put((size_t)J * 4);
  c.H1 = put((size_t)nb * 4);
  c.VH1 = put((size_t)nb * 12);
  c.VL1 = put((size_t)nb * 12);
  c.W2 = put(nw * 32 * kDenseGroup * 4);
  c.Val = put(nw * kDenseCap * 4);
  c.Ent = put(nw * kDenseCap * 2);
  c.KLs = put((na * na + 1) * 4);
  c.KLg = put((size_t)G * 4);
  c.Mult = put((size_t)J);
  c.total = o;
  return c;
}

// NB complex floats from shared memory, 16 bytes at a time where the row length allows
template <int NB>
__device__ __forceinline__ void ld_row(const Cx<float>* p, Cx<float>* out) {
  if constexpr (NB % 2 == 0) {
#pragma unroll
    for (int i = 0; i < NB / 2; ++i) {
      const float4 v = reinterpret_cast<const float4*>(p)[i];
      out[2 * i] = cmk<float>(v.x, v.y);
      out[2 * i + 1] = cmk<float>(v.z, v.w);
    }
  } else {
#pragma unroll
    for (int i = 0; i < NB; ++i) out[i] = p[i];
  }
}

// a + b of two-float numbers, rounded to FP32 (error 2^-24 of the result and about 2^-46 of the operands)
__device__ __forceinline__ float sum2(float ah, float al, float bh, float bl) {
  float s, e;
  two_sum(ah, bh, s, e);
  return s + (e + (al + bl));
}

// the Gaussian times 1/sigma, or 1 where delta := 1 (inv < 0), by the operations of fp_rates_kernel.cuh
__device__ __forceinline__ float delta_f32(float dw, float inv) {
  const float xx = dw * inv;
  const float d = __expf(-xx * xx) * inv * (float)kInvSqrtPi;
  return inv >= 0.f ? d : 1.0f;
}

// FP64 decision of candidate c of the entry, in the operation order of the definition
__device__ __noinline__ bool dense_decide(const RatesArgs& a, int c, int q0, int k1x, int k2y, int k3j) {
  const bool ordA = c < 3;
  const double* vl = a.vel + 3 * (size_t)(ordA ? k2y : k1x);
  double ex[2];
  sigma_entry(a, vl, (c == 0 || c == 3) ? 1.0 : -1.0, a.vel + 3 * (size_t)k3j, ex);
  return fabs(dw_fp64(c, a.omega[q0], a.omega[k1x], a.omega[k2y], a.omega[k3j])) <= ex[0];
}

template <int NB, int MAXT>
__global__ void __launch_bounds__(max_threads_for(NB), dense_blocks_for(NB)) dense_kernel(RatesArgs a) {
  constexpr int NB2 = NB * NB, NA = NB / 3, kAB = NB2 + 2, kUn = MAXT == 1 ? kDenseGroup : 2;
  using C = Cx<float>;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ long long s_item;
  __shared__ unsigned s_umask[2];
  const int J = a.J, G = a.G, nT = MAXT == 1 ? 1 : a.nT, N = a.N;
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const int rows = J * NB2;
  const DenseCarve cv = make_dense_carve(NB, J, G, a.nquart, nT, nthr);
  const DenseRecord rd = make_record(NB, G, nT);
  auto cxp = [&](size_t at) { return reinterpret_cast<C*>(smem + at); };
  auto flt = [&](size_t at) { return reinterpret_cast<float*>(smem + at); };
  auto flt2 = [&](size_t at) { return reinterpret_cast<float2*>(smem + at); };
  auto flt4 = [&](size_t at) { return reinterpret_cast<float4*>(smem + at); };
  C *sE0 = cxp(cv.E0), *sE1 = cxp(cv.E1), *sPsi = cxp(cv.Psi), *sTwQ = cxp(cv.TwQ), *sA = cxp(cv.A);
  double* sRed = reinterpret_cast<double*>(smem + cv.A);
  float *sRec = flt(cv.Rec), *sF0 = flt(cv.F0), *sH0 = flt(cv.H0), *sH1 = flt(cv.H1), *sVH1 = flt(cv.VH1), *sVL1 = flt(cv.VL1);
  float4 *sX = flt4(cv.X), *sT1 = flt4(cv.T1), *sT3 = flt4(cv.T3), *sU = flt4(cv.U);
  float2 *sT0 = flt2(cv.T0), *sT2 = flt2(cv.T2), *sF1 = flt2(cv.F1);
  float* sW2 = flt(cv.W2) + warp * 32 * kDenseGroup;
  float* sVal = flt(cv.Val) + warp * kDenseCap;
  unsigned short* sEnt = reinterpret_cast<unsigned short*>(smem + cv.Ent) + warp * kDenseCap;
  int *sKLs = reinterpret_cast<int*>(smem + cv.KLs), *sKLg = reinterpret_cast<int*>(smem + cv.KLg);
  unsigned char* sMult = smem + cv.Mult;

  const bool has_row = tid < rows;
  const int rjj = has_row ? tid / NB2 : 0, rj1 = has_row ? (tid / NB) % NB : 0, rc = tid % NB;
  const int ab = rjj * NB + rj1;
  const size_t NM = (size_t)N * NB;
  const bool f32_sigma = a.dq_mode == 0;
  const bool unit = a.unit_vertex != 0;

  for (int o = tid; o < NA * NA + 1; o += nthr) sKLs[o] = a.kl_start[o];
  for (int o = tid; o < G; o += nthr) sKLg[o] = a.kl_grp[o];

  for (;;) {
    __syncthreads();  // the tables above; at later items, the last epilogue's reads
    if (tid == 0) s_item = (long long)atomicAdd(a.counter, 1ULL);
    __syncthreads();
    const long long item = s_item;
    if (item >= a.n_items) break;
    const int chunk = (int)(item % a.nchunk);
    const long long rest = item / a.nchunk;
    const int qi = (int)(rest % a.nq_sel);
    const int tile = (int)(rest / a.nq_sel);
    const int q = a.qlist[qi];
    const int j0b = chunk * J;
    const int g[3] = {q / (a.grid[1] * a.grid[2]), (q / a.grid[2]) % a.grid[1], q % a.grid[2]};
    for (int o = tid; o < J * NB; o += nthr) sE0[o] = ld_e<float>(a, ((size_t)q * NB + j0b) * NB + o);
    for (int jj = tid; jj < J; jj += nthr) {
      const int m = q * NB + j0b + jj;
      sH0[jj] = a.omh[m];
      sMult[jj] = a.omega[m] > 0.0 ? a.mult[m] : 0;
    }
    for (int o = tid; o < nT * J; o += nthr) sF0[o] = a.wtf[3 * ((size_t)(o / J) * NM + (size_t)q * NB + j0b + o % J)];
    __syncthreads();
    int any = 0;
    float hm0 = 0.f;
    for (int jj = 0; jj < J; ++jj) {
      any |= sMult[jj];
      hm0 = fmaxf(hm0, sH0[jj]);
    }
    const unsigned row_mult = has_row ? sMult[rjj] : 0u;

    float acch[MAXT], accl[MAXT];
#pragma unroll
    for (int t = 0; t < MAXT; ++t) acch[t] = accl[t] = 0.f;
    auto comp = [&](int t, float v) {
      float s, e;
      two_sum(acch[t], v, s, e);
      acch[t] = s;
      accl[t] += e;
    };
    unsigned n0 = 0, n1 = 0, n2 = 0, it = 0;  // accepted terms of the row per process; k2 steps
    const int k1_begin = tile * a.t1;
    const int k1_end = min(N, k1_begin + a.t1);
    const int k1_first = unit ? ((k1_begin + a.k1_stride - 1) / a.k1_stride) * a.k1_stride : k1_begin;
    const int k1_step = unit ? a.k1_stride : 1;
    for (int k1 = any ? k1_first : k1_end; k1 < k1_end; k1 += k1_step) {
      const int g1[3] = {k1 / (a.grid[1] * a.grid[2]), (k1 / a.grid[2]) % a.grid[1], k1 % a.grid[2]};
      __syncthreads();  // the last k1's reads
      for (int o = tid; o < NB2; o += nthr) sE1[o] = ld_e<float>(a, (size_t)k1 * NB2 + o);
      for (int o = tid; o < NB; o += nthr) sH1[o] = a.omh[k1 * NB + o];
      for (int o = tid; o < 3 * NB; o += nthr) {
        sVH1[o] = a.velh[(size_t)k1 * NB * 3 + o];
        sVL1[o] = a.vell[(size_t)k1 * NB * 3 + o];
      }
      for (int o = tid; o < nT * NB; o += nthr) {
        const float* w = a.wtf + 3 * ((size_t)(o / NB) * NM + (size_t)k1 * NB + o % NB);
        sF1[o] = make_float2(w[1], w[2]);
      }
      for (int o = tid; o < J * NB; o += nthr) {
        const double w0 = a.omega[q * NB + j0b + o / NB], w1 = a.omega[k1 * NB + o % NB];
        const float2 s = df_make(w0 + w1), d = df_make(w0 - w1);
        sX[o] = make_float4(s.x, s.y, d.x, d.y);
      }
      if (!unit)
        for (int Q = tid; Q < a.nquart; Q += nthr) {
          const int* m = a.qmeta + 9 * Q;
          int e = 0;  // each term is below L, so e < 3 L
          for (int d = 0; d < 3; ++d) e += a.Lfac[d] * wrapi(g1[d] * m[3 + d] - (g[d] + g1[d]) * m[6 + d], a.grid[d]);
          while (e >= a.L) e -= a.L;
          sTwQ[Q] = ld_tw<float>(a, e);
        }
      __syncthreads();
      float hm1 = 0.f;
      for (int x = 0; x < NB; ++x) hm1 = fmaxf(hm1, sH1[x]);
      if (!unit) {
        // products e0(i alpha) e1(j beta) of every (j0, x), then Psi[jj][j1][grp][gt] as in fp_rates_kernel.cuh
        for (int o = tid; o < J * NB * NB2; o += nthr) {
          const int jr = o / NB2, c0 = (o / NB) % NB, c1 = o % NB;
          sA[(size_t)jr * kAB + c0 * NB + c1] = cmul(sE0[(jr / NB) * NB + c0], sE1[(jr % NB) * NB + c1]);
        }
        __syncthreads();
        constexpr int kGtb = 3;
        for (int o = tid; o < J * NB * G * (9 / kGtb); o += nthr) {
          const int gb = o % (9 / kGtb), jr = (o / (9 / kGtb)) % (J * NB), grp = o / ((9 / kGtb) * J * NB);
          C sum[kGtb];
#pragma unroll
          for (int u = 0; u < kGtb; ++u) sum[u] = cmk<float>(0, 0);
          for (int qq = a.grp_qstart[grp]; qq < a.grp_qstart[grp + 1]; ++qq) {
            const int Q = a.grp_q[qq];
            const C* pr = sA + (size_t)jr * kAB + 3 * a.qmeta[9 * Q] * NB + 3 * a.qmeta[9 * Q + 1];
            const C tq = sTwQ[Q];
            const float* fc = a.qfcf + 81 * (size_t)Q + gb * kGtb;
            C s[kGtb];
#pragma unroll
            for (int u = 0; u < kGtb; ++u) s[u] = cmk<float>(0, 0);
#pragma unroll
            for (int p = 0; p < 9; ++p) {
              const C pv = pr[(p / 3) * NB + p % 3];
#pragma unroll
              for (int u = 0; u < kGtb; ++u) {
                const float fv = fc[p * 9 + u];
                s[u].re = fmaf(fv, pv.re, s[u].re);
                s[u].im = fmaf(fv, pv.im, s[u].im);
              }
            }
#pragma unroll
            for (int u = 0; u < kGtb; ++u) cfma(sum[u], tq, s[u]);
          }
#pragma unroll
          for (int u = 0; u < kGtb; ++u) sPsi[(size_t)(jr * G + grp) * 9 + gb * kGtb + u] = sum[u];
        }
      }

      // the records of (k2, k3), one step ahead: 16 bytes per thread in registers until the buffer is free
      const int gs[3] = {(g[0] + g1[0]) % a.grid[0], (g[1] + g1[1]) % a.grid[1], (g[2] + g1[2]) % a.grid[2]};
      int k2 = unit ? 0 : k1;
      int g2[3] = {k2 / (a.grid[1] * a.grid[2]), (k2 / a.grid[2]) % a.grid[1], k2 % a.grid[2]};
      auto third = [&]() {
        int k3 = 0;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          int x = gs[d] + g2[d];
          if (x >= a.grid[d]) x -= a.grid[d];
          k3 = k3 * a.grid[d] + x;
        }
        return k3;
      };
      const int nrec4 = rd.size / 2, half = rd.size / 4;
      constexpr int kPre = NB == 6 || (NB == 3 && MAXT == 1) ? 1 : 2;
      float4 pre[kPre];
      int k3 = third();
      auto fetch = [&]() {
#pragma unroll
        for (int p = 0; p < kPre; ++p) {
          const int o = tid + p * nthr;
          if (o < nrec4)
            pre[p] = reinterpret_cast<const float4*>(a.rec32 + (size_t)(o < half ? k2 : k3) * rd.size)[o < half ? o : o - half];
        }
      };
      fetch();
      __syncthreads();  // Psi complete, the products in sA read
      for (int buf = 0; k2 < N; buf ^= 1) {
        {
          float4* dst = reinterpret_cast<float4*>(sRec + (size_t)buf * 2 * rd.size);
#pragma unroll
          for (int p = 0; p < kPre; ++p)
            if (tid + p * nthr < nrec4) dst[tid + p * nthr] = pre[p];
          for (int o = tid + kPre * nthr; o < nrec4; o += nthr)
            dst[o] = reinterpret_cast<const float4*>(a.rec32 + (size_t)(o < half ? k2 : k3) * rd.size)[o < half ? o : o - half];
          if (a.nu_select != 0 && tid == 0) {
            const int g3[3] = {k3 / (a.grid[1] * a.grid[2]), (k3 / a.grid[2]) % a.grid[1], k3 % a.grid[2]};
            s_umask[buf] = umklapp_bits(a, g, g1, g2, g3);
          }
        }
        const int c2 = k2, c3 = k3;
        __syncthreads();  // the records are in place; the last k2's A and tables have been read
        if (++k2 < N) {
          if (++g2[2] == a.grid[2]) {
            g2[2] = 0;
            if (++g2[1] == a.grid[1]) {
              g2[1] = 0;
              ++g2[0];
            }
          }
          k3 = third();
          fetch();
        }
        const float* r2 = sRec + (size_t)buf * 2 * rd.size;
        const float* r3 = r2 + rd.size;
        // ---- tables: [y][j3] of v(k2, y) and of the sums with w(k2, y), [x][j3] of v(k1, x)
        for (int o = tid; o < 2 * NB2; o += nthr) {
          const bool of1 = o >= NB2;
          const int e = of1 ? o - NB2 : o, u = e / NB, j3 = e % NB;
          const float *vh = of1 ? sVH1 + 3 * u : r2 + rd.VH + 3 * u, *vl = of1 ? sVL1 + 3 * u : r2 + rd.VL + 3 * u;
          const double *v64 = a.vel + 3 * ((size_t)(of1 ? k1 : c2) * NB + u), *v364 = a.vel + 3 * ((size_t)c3 * NB + j3);
          float2 pm[2];
          float inv[2];
#pragma unroll
          for (int s = 0; s < 2; ++s) {
            if (f32_sigma) {
              sigma_entry_f32(a, vh, vl, s ? -1.f : 1.f, r3 + rd.VH + 3 * j3, r3 + rd.VL + 3 * j3, v64, v364, &pm[s], &inv[s]);
            } else {
              double ex[2];
              sigma_entry(a, v64, s ? -1.0 : 1.0, v364, ex);
              sigma_f_from_exact(ex, &pm[s], &inv[s]);
            }
          }
          const float h3 = r3[rd.H + j3];
          float hsum = hm0 + h3;  // an upper bound of the entry's frequency sum, for the prefilter's margin
          if (of1) {
            float hm2 = 0.f;
            for (int y = 0; y < NB; ++y) hm2 = fmaxf(hm2, r2[rd.H + y]);
            hsum += sH1[u] + hm2;
          } else {
            hsum += hm1 + r2[rd.H + u];
          }
          const float m = 1.001f * kRelS * hsum;
          (of1 ? sT3 : sT1)[e] = make_float4(pm[1].x - (m + pm[1].y), pm[1].x + (m + pm[1].y), inv[1], pm[0].x + (m + pm[0].y));
          (of1 ? sT2 : sT0)[e] = make_float2(pm[0].x - (m + pm[0].y), inv[0]);
          if (!of1) {
            const float hy = r2[rd.H + u], ly = r2[rd.L + u], l3 = r3[rd.L + j3];
            float s1, e1, s2, e2;
            two_sum(hy, h3, s1, e1);
            two_sum(hy, -h3, s2, e2);
            const float2 p = df_fast(s1, e1 + (ly + l3)), n = df_fast(s2, e2 + (ly - l3));
            const float nan = __int_as_float(0x7fffffff);
            sU[e] = hy != 0.f && h3 != 0.f ? make_float4(p.x, p.y, n.x, n.y) : make_float4(nan, nan, nan, nan);
          }
        }
        if (has_row && !unit) {
          // A row of component rc = (ka, ga): one pass over the groups of atom ka, which sit contiguously in l order
          const int ka = rc / 3, ga = rc % 3;
          const C* psi_row = sPsi + (size_t)ab * G * 9 + ga * 3;
          const C* tw2 = reinterpret_cast<const C*>(r2 + rd.Tw);
          C* arow = sA + (size_t)ab * kAB + rc * NB;
          int gi = sKLs[ka * NA];
#pragma unroll
          for (int l = 0; l < NA; ++l) {
            const int seg_end = sKLs[ka * NA + l + 1];
            C cur[3] = {cmk<float>(0, 0), cmk<float>(0, 0), cmk<float>(0, 0)};
            for (; gi < seg_end; ++gi) {
              const int grp = sKLg[gi];
              const C tw = tw2[grp];
              const C* ps = psi_row + grp * 9;
#pragma unroll
              for (int th = 0; th < 3; ++th) cfma(cur[th], tw, ps[th]);
            }
#pragma unroll
            for (int th = 0; th < 3; ++th) arow[3 * l + th] = cur[th];
          }
        }
        __syncthreads();
        // ---- column j3 = rc of T; per y: W, tests, the +- terms
        const unsigned cand = (row_mult ? 0x3Fu : 0u) & ((k1 != c2 && !unit) ? 0x3Fu : 0x07u) & a.cand_mask &
                              (a.nu_select == 0 ? 0x3Fu : a.nu_select == 1 ? ~s_umask[buf] : s_umask[buf]);
        C T[NB];
        if (!unit && has_row) {
          C e3[NB], row[NB];
          ld_row<NB>(reinterpret_cast<const C*>(r3 + rd.E) + rc * NB, e3);
#pragma unroll
          for (int k = 0; k < NB; ++k) {
            ld_row<NB>(sA + (size_t)ab * kAB + k * NB, row);
            T[k] = cmk<float>(0, 0);
#pragma unroll
            for (int d = 0; d < NB; ++d) cfma_conj(T[k], row[d], e3[d]);
          }
        }
        const float4 X = sX[ab], t3 = sT3[rj1 * NB + rc];
        const float2* w2v = reinterpret_cast<const float2*>(r2 + rd.W);
        const float2* w3v = reinterpret_cast<const float2*>(r3 + rd.W);
        const bool xok = sH1[rj1] != 0.f;
        const bool c1ok = xok && (cand & 2u), c4ok = xok && (cand & 16u);
        const unsigned rare = xok ? cand & 0x2Du : 0u;
        float f0h = 0.f, a1 = 0.f, b1 = 0.f, F3 = 0.f;
        if constexpr (MAXT == 1) {
          f0h = 0.5f * sF0[rjj];
          a1 = sF1[rj1].x;
          b1 = sF1[rj1].y;
          F3 = w3v[rc].y;
        }
#pragma unroll 1
        for (int jb = 0; jb < NB; jb += kDenseGroup) {
          constexpr int kG = NB < kDenseGroup ? NB : kDenseGroup;
          unsigned m = 0;  // accepted candidates 0, 2, 3, 5: bit kind * kDenseGroup + u
#pragma unroll kUn
          for (int u = 0; u < kG; ++u) {
            const int y = jb + u, e = y * NB + rc;
            float w2 = 1.f;
            if (!unit) {
              C e2[NB];
              ld_row<NB>(reinterpret_cast<const C*>(r2 + rd.E) + y * NB, e2);
              C Wv = cmk<float>(0, 0);
#pragma unroll
              for (int c = 0; c < NB; ++c) cfma(Wv, e2[c], T[c]);
              w2 = Wv.re * Wv.re + Wv.im * Wv.im;
            }
            const float4 t1 = sT1[e], U = sU[e];
            const float dw1 = sum2(X.x, X.y, -U.x, -U.y), dw4 = sum2(X.z, X.w, U.z, U.w);
            const float ad1 = fabsf(dw1), ad4 = fabsf(dw4);
            bool in1 = c1ok && ad1 < t1.x, in4 = c4ok && ad4 < t3.x;
            const bool b1nd = c1ok && ad1 <= t1.y && !(ad1 < t1.x), b4nd = c4ok && ad4 <= t3.y && !(ad4 < t3.x);
            const float d03 = fabsf(X.x + U.z), d25 = fabsf(X.z - U.x);
            if (b1nd | b4nd | (rare && (d03 <= fmaxf(t1.w, t3.w) || d25 <= fmaxf(t1.y, t3.y)))) {
              const int q0 = q * NB + j0b + rjj, kx = k1 * NB + rj1, ky = c2 * NB + y, kj = c3 * NB + rc;
              if (b1nd) in1 = dense_decide(a, 1, q0, kx, ky, kj);
              if (b4nd) in4 = dense_decide(a, 4, q0, kx, ky, kj);
              const float2 t0 = sT0[e], t2 = sT2[rj1 * NB + rc];
              unsigned acc = (d03 < t0.x ? 1u : 0u) | (d25 < t1.x ? 4u : 0u) | (d03 < t2.x ? 8u : 0u) | (d25 < t3.x ? 32u : 0u);
              unsigned band = (d03 <= t1.w ? 1u : 0u) | (d25 <= t1.y ? 4u : 0u) | (d03 <= t3.w ? 8u : 0u) | (d25 <= t3.y ? 32u : 0u);
              band &= rare & ~acc;
              acc &= rare;
              for (; band; band &= band - 1)
                if (dense_decide(a, __ffs(band) - 1, q0, kx, ky, kj)) acc |= band & (0u - band);
              // candidates 0, 2, 3, 5 to bits 0, 6, 12, 18
              acc = (acc & 1u) | (acc & 4u) << (kDenseGroup - 2) | (acc & 8u) << (2 * kDenseGroup - 3) |
                    (acc & 32u) << (3 * kDenseGroup - 5);
              if (acc) {
                m |= acc << u;
                sW2[u * 32 + lane] = w2;  // waits for the compacted evaluation below
              }
            }
            n1 += (in1 ? 1u : 0u) + (in4 ? 1u : 0u);
            const float wd1 = delta_f32(dw1, t1.z), wd4 = delta_f32(dw4, t3.z);
            if constexpr (MAXT == 1) {
              const float2 f2 = w2v[y];
              const float v1 = (w2 * wd1) * (f0h * (a1 * f2.y)) * F3, v4 = (w2 * wd4) * (f0h * (f2.x * b1)) * F3;
              comp(0, in1 ? v1 : 0.f);
              comp(0, in4 ? v4 : 0.f);
            } else {
              const float base1 = 0.5f * w2 * wd1, base4 = 0.5f * w2 * wd4;
              if (in1 | in4) {
#pragma unroll
                for (int t = 0; t < MAXT; ++t) {
                  if (t >= nT) break;
                  const float f0 = sF0[t * J + rjj], f3 = w3v[t * NB + rc].y;
                  const float2 f1 = sF1[t * NB + rj1], f2 = w2v[t * NB + y];
                  const float v1 = base1 * f0 * f1.x * f2.y * f3, v4 = base4 * f0 * f2.x * f1.y * f3;
                  comp(t, in1 ? v1 : 0.f);
                  comp(t, in4 ? v4 : 0.f);
                }
              }
            }
          }
          // the other accepted candidates of the warp, compacted in lane order and evaluated 32 at a time
          if (__any_sync(0xffffffffu, m != 0)) {
            constexpr unsigned kM = (1u << kDenseGroup) - 1u;
            n0 += __popc(m & (kM | kM << (2 * kDenseGroup)));
            n2 += __popc(m & (kM << kDenseGroup | kM << (3 * kDenseGroup)));
            const int nmy = __popc(m);
            int incl = nmy;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const int v = __shfl_up_sync(0xffffffffu, incl, o);
              if (lane >= o) incl += v;
            }
            const int total = __shfl_sync(0xffffffffu, incl, 31);
            int pos = incl - nmy;
            unsigned left = m;
            for (int r0 = 0; r0 < total; r0 += kDenseCap) {
              const int rn = min(total - r0, kDenseCap);
              const int pos0 = pos;
              const unsigned left0 = left;
              for (; left && pos < r0 + kDenseCap; left &= left - 1)
                sEnt[pos++ - r0] = (unsigned short)(lane | (__ffs(left) - 1) << 5);
              __syncwarp();
              for (int i = lane; i < rn; i += 32) {
                const unsigned en = sEnt[i];
                const int src = (int)(en & 31u), row = (tid & ~31) + src, bit = (int)(en >> 5);
                const int kind = bit / kDenseGroup, u = bit % kDenseGroup, y = jb + u, j3 = row % NB;
                const int ej = row / NB2, ex = (row / NB) % NB, e = y * NB + j3, e1 = ex * NB + j3;
                const float4 Xe = sX[row / NB], Ue = sU[e];
                const bool plus = kind == 0 || kind == 2;
                const float dw = plus ? sum2(Xe.x, Xe.y, Ue.z, Ue.w) : sum2(Xe.z, Xe.w, -Ue.x, -Ue.y);
                const float inv = kind == 0 ? sT0[e].y : kind == 1 ? sT1[e].z : kind == 2 ? sT2[e1].y : sT3[e1].z;
                const float w2 = sW2[u * 32 + src], delta = delta_f32(dw, inv);
                float v;
                if constexpr (MAXT == 1) {
                  const float f0 = sF0[ej];
                  const float2 f1 = sF1[ex], f2 = w2v[y];
                  const float wsel = plus ? 0.5f * f0 * (f1.x * f2.x) : (1.0f / 6.0f) * f0 * (f1.y * f2.y);
                  v = (w2 * delta) * wsel * w3v[j3].y;
                } else {
                  v = (plus ? 0.5f : 1.0f / 6.0f) * w2 * delta;
                }
                sVal[i] = v;
              }
              __syncwarp();
              int p = pos0 - r0;
              for (unsigned b = left0 & ~left; b; b &= b - 1) {
                const int bit = __ffs(b) - 1, kind = bit / kDenseGroup, y = jb + bit % kDenseGroup;
                const float v = sVal[p++];
                if constexpr (MAXT == 1) {
                  comp(0, v);
                } else {
                  const bool plus = kind == 0 || kind == 2;
#pragma unroll
                  for (int t = 0; t < MAXT; ++t) {
                    if (t >= nT) break;
                    const float2 f1 = sF1[t * NB + rj1], f2 = w2v[t * NB + y];
                    const float x1 = plus ? f1.x : f1.y, x2 = plus ? f2.x : f2.y;
                    comp(t, v * sF0[t * J + rjj] * (kind < 2 ? x1 : x2) * (kind < 2 ? x2 : x1) * w3v[t * NB + rc].y);
                  }
                }
              }
              __syncwarp();
            }
          }
        }
        ++it;
      }
    }
    // rows of each j0 in order
    __syncthreads();
    if (has_row) {
#pragma unroll
      for (int t = 0; t < MAXT; ++t) {
        if (t >= nT) break;
        sRed[(size_t)tid * nT + t] = (double)acch[t] + (double)accl[t];
      }
    }
    __syncthreads();
    for (int o = tid; o < J * nT; o += nthr) {
      const int jj = o / nT, t = o % nT;
      double sum = 0.0;
      for (int r = 0; r < NB2; ++r) sum += sRed[(size_t)(jj * NB2 + r) * nT + t];
      a.partial[(size_t)item * J * nT + o] = sum;
    }
    __syncthreads();
    const unsigned nte = n0 + n1 + n2;
    if (a.item_counts) {
      // accepted terms per j0 of the item, in row order
      unsigned long long* sCnt = reinterpret_cast<unsigned long long*>(sRed);
      sCnt[tid] = nte;
      __syncthreads();
      for (int jj = tid; jj < J; jj += nthr) {
        unsigned long long sum = 0;
        for (int r = jj * NB2; r < (jj + 1) * NB2; ++r) sum += sCnt[r];
        a.item_counts[(size_t)item * J + jj] = sum;
      }
      __syncthreads();
    }
    const unsigned long long mult = row_mult;
    unsigned long long c0 = mult * n0, c1 = mult * n1, c2 = mult * n2, ct = nte;
    unsigned long long cw = !unit && row_mult ? (unsigned long long)it * NB : 0ull;
    for (int off = 16; off > 0; off >>= 1) {
      c0 += __shfl_down_sync(0xffffffffu, c0, off);
      c1 += __shfl_down_sync(0xffffffffu, c1, off);
      c2 += __shfl_down_sync(0xffffffffu, c2, off);
      cw += __shfl_down_sync(0xffffffffu, cw, off);
      ct += __shfl_down_sync(0xffffffffu, ct, off);
    }
    if (lane == 0) {
      if (c0) atomicAdd(a.counts + 0, c0);
      if (c1) atomicAdd(a.counts + 1, c1);
      if (c2) atomicAdd(a.counts + 2, c2);
      if (cw) atomicAdd(a.counts + 3, cw);
      if (ct) atomicAdd(a.counts + 4, ct);
    }
  }
}

}  // namespace
}  // namespace fp

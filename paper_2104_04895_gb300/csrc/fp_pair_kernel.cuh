// Four-phonon rate kernel over unordered wavevector pairs (FP64 and double-float paths; paper Sec. 2.2 Eqs. tao0,
// 4phgamma, V4; Sec. 2.4).  Used when the quartet list obeys the transposition symmetry of Sec. 2.3 (Eq. TS), which
// fp_init checks; otherwise the kernel of fp_rates_kernel.cuh runs.  One pass can keep the parts of a rate apart
// (RatesArgs::split): normal and Umklapp processes, which one k2 decides for a whole test, or the three channels.
//
// What it shares.  The rate of a = (q, j0) is a sum over b = lambda' of R(a; b), where R(a; b) collects every process
// in which b is the partner lambda' and {c, d} are lambda'', lambda''' in both orders.  Write all four wavevectors as
// incoming (q + k1 + k2 + kd = 0, so kd = -k3 with the k3 = q + k1 + k2 of fp_rates_kernel.cuh).  The broadening
// |v'' - v'''| of Sec. 2.4 then depends on c and d alone, so for one entry (a, b, c, d) five energy tests cover it:
//   P1  wa + wb - wc - wd   +- with lambda'' = c or d (two orders)       -> R(a; b) and R(b; a)
//   P2  wa + wb + wc - wd   ++ with lambda'' = c                         -> R(a; b) and R(b; a)
//   P3  wa + wb + wd - wc   ++ with lambda'' = d                         -> R(a; b) and R(b; a)
//   P4  wa - wb - wc - wd   -- of a (two orders)                          -> R(a; b)
//   P5  wb - wa - wc - wd   -- of b (two orders)                          -> R(b; a)
// with sigma = |v(k2) - v(k3)| for P2, P3 and |v(k2) + v(k3)| for P1, P4, P5.  One vertex W and, for P1 (nearly all
// accepted terms), one Gaussian serve four terms of the ordered sum; the loop over k2 stops at k2 <= kd, and a pair
// {a, b} is visited once when both a and b (or -b) are evaluated points.  Against the kernel that visits every
// ordered q' this halves the vertices and quarters the window tests and Gaussians.
// The leg weights of a and b leave the inner sum: with S1 = sum over P1, P2, P3 of |W|^2 delta x (c and d weights),
// S4 and S5 likewise,
//   R(a; b) = f0(a) [ (1 + nb)/wb S1 + nb/wb S4 ],   R(b; a) = f0(b) [ (1 + na)/wa S1 + na/wa S5 ],   f0 = 1/(n w).
// With x = hbar w / k_B T the product nc nd inside goes as exp(-(xc + xd)), xc + xd about xa + xb, and f0 as exp(xa): at low
// temperature the product underflows where the rate, about exp(-xb), does not.  So the c and d weights carry a power of
// two each, near exp(x/2) of the largest frequency, and f0 carries its inverse square: the products then stay between
// exp(-x) and exp(x), and every bit is as without it where the plain product is a normal number.
//
// Both values go to their own slot of `partial` ([evaluated point][partner b]); pair_reduce_kernel sums the slots of a
// mode in a fixed order.  No atomics touch the rates.
//
// Thread r < J nb^2 owns the row (j0, x = branch of b, y = branch of c): it builds the A and T rows (j0, x, component
// y), screens its nb entries and accumulates their terms.  The accepted (entry, test) pairs of a warp's 32 rows are
// compacted into a list that the warp evaluates 32 at a time (W, Gaussian), and each value returns to the row that
// owns it: the FP64 pipe, the bound of the FP64 path, runs on full warps however unevenly the terms fall on rows.
//
// On the FP64 path with 6 or 12 branches and unit eigenvectors both vertex contractions run on the tensor cores in exact
// integer slices (SL, fp_slices.cuh): A is built in FP64, its digits contract with those of e3 to T, T's digits with those of e2 to
// every W of the block, which costs the FP64 pipe only the A sums and |W|^2.  A scale per (j0, x), the power of two
// above the Frobenius norm of its A block, keeps all three in range.  Terms whose W is below 2^-12 of that scale are
// bounded a second time at the scale itself (sWeak, a.weak), from which the reduction sees the rates that need the FP64
// contraction (fp_slices.cuh).
//
// Measured (GB300): ordered kernel -> pair kernel -> with slices and the U table of the prologue -> with U over terms and
// several items per pair on small grids:
//   diamond 6^3 FP64            578 -> 223 -> 125 -> 120 ms      LiCoO2 5x4x3 FP64, 3 T   386 -> 154 -> 82 -> 77 ms
//   diamond 7x6x5 double-float  262 -> 88 -> 87 -> 91 ms (no slices: 107 ms with them, the FP64 A sums and conversions
//                               cost more than the FP32 contraction; LiCoO2 4x3x3 24.3 ms either way)
//   simple cubic 4^3 FP64       2.15 -> 1.49 -> 1.13 -> 0.91 ms (nb = 3: no slices)
// The last double-float step evaluates the accepted terms in FP64 (before, in pairs of floats, whose weights underflowed
// below about 20 K): 87 -> 91 ms with one temperature, 106 -> 103 with three, 126 -> 119 with eight, LiCoO2 4x3x3 17.2 ->
// 16.8 and 22.3 -> 20.0 with three.
// Without slices the FP64 pipe (about 1.7 lane FMAs per clock and SM) is 91 % busy: per k2 of six branches 31k lane
// FMAs for T, 20k for W, 8k for A, 12k for the terms.  With them it is 68 % busy (diamond 4^3), three quarters of that
// with the terms (20 instructions each), the rest with A; the barriers between the phases cost most of the other 32 %.
#pragma once
#include "fp_rates_kernel.cuh"
#include "fp_slices.cuh"

namespace fp {
namespace {

constexpr int kPairGroup = 6;   // j3 values compacted at once (five tests each: 30 bits of a lane's mask)
constexpr int kPairCap = 128;   // list entries per warp and round

// Role of the slot (qi, b) of `partial`: the value R(q; b) of the evaluated point q = qlist[qi].
struct PairRole {
  bool run;     // evaluate the pair (q, b) here
  int mirror;   // evaluated-point index whose slot (mirror, mirror_b) takes R(b; q), or -1
  int mirror_b;
};

__device__ __forceinline__ int neg_q(const RatesArgs& a, int q) {
  const int g0 = q / (a.grid[1] * a.grid[2]), g1 = (q / a.grid[2]) % a.grid[1], g2 = q % a.grid[2];
  const int m0 = g0 ? a.grid[0] - g0 : 0, m1 = g1 ? a.grid[1] - g1 : 0, m2 = g2 ? a.grid[2] - g2 : 0;
  return (m0 * a.grid[1] + m1) * a.grid[2] + m2;
}

// A pair {q, b} with b = s r (r an evaluated point, s = +1 or -1 by time reversal) holds two wanted values: R(q; b) in
// the slot (q, b) and R(b; q) = R(r; s q) in the slot (r, s q).  The one with the smaller evaluated index runs and
// writes both.  A self-conjugate q with s = -1 would share its mirror slot with (q, r), so it runs by itself.
__device__ __forceinline__ PairRole pair_role(const RatesArgs& a, int qi, int q, int b) {
  PairRole p;
  p.run = true;
  p.mirror = -1;
  p.mirror_b = 0;
  if (!a.mirror) return p;
  const int ri = a.qpos[b];
  if (ri < 0 || ri == qi) return p;
  const bool plus = a.qlist[ri] == b;
  const int nq = plus ? q : neg_q(a, q);
  if (!plus && nq == q) return p;
  if (qi < ri) {
    p.mirror = ri;
    p.mirror_b = nq;
  } else {
    p.run = false;
  }
  return p;
}

// Umklapp classes of one (q, k1, k2) pair entry, bits 0..4 for P1..P5 (Q of Sec. 2.2 with every wavevector as its
// Brillouin-zone representative g / N - m).
__device__ unsigned pair_umklapp_bits(const RatesArgs& a, const int g[3], const int g1[3], const int g2[3],
                                      const int g3[3]) {
  // k x representative of grid point x (sign +1) or of its negative (sign -1), integer numerators
  auto rep = [&](const int* x, int sign, int d) {
    int y[3];
    for (int e = 0; e < 3; ++e) y[e] = sign > 0 ? x[e] : (x[e] ? a.grid[e] - x[e] : 0);
    const int i = (y[0] * a.grid[1] + y[1]) * a.grid[2] + y[2];
    return y[d] - a.grid[d] * a.bzm[3 * i + d];
  };
  unsigned u = 0;
  for (int d = 0; d < 3; ++d) {
    const int ra = rep(g, 1, d), rb = rep(g1, 1, d), rc = rep(g2, 1, d), r3 = rep(g3, 1, d);
    const int na = rep(g, -1, d), nb = rep(g1, -1, d), nc = rep(g2, -1, d), n3 = rep(g3, -1, d);
    u |= (ra + rb - nc - r3 != 0) ? 1u : 0u;   // P1: a + b -> c', d'  (c' = -k2, d' = k3)
    u |= (ra + rb + rc - r3 != 0) ? 2u : 0u;   // P2: a + b + c -> d'
    u |= (ra + rb + n3 - nc != 0) ? 4u : 0u;   // P3: a + b + d -> c'  (d = -k3)
    u |= (ra - nb - nc - r3 != 0) ? 8u : 0u;   // P4: a -> b' + c' + d'
    u |= (rb - na - nc - r3 != 0) ? 16u : 0u;  // P5: b -> a' + c' + d'
  }
  return u;
}

// Largest block (rows of two j0 for twelve branches: one block of nine warps fills the shared memory of an SM, where
// one j0 would leave room for one block of five; two blocks per SM otherwise).
__host__ __device__ constexpr int pair_threads_for(int nb) { return nb == 12 ? 288 : max_threads_for(nb); }
__host__ __device__ constexpr int pair_blocks_for(int nb) { return nb == 12 ? 1 : 2; }

struct PairCarve {
  size_t E0, E1, E2, E3, Psi, T, Tw2, TwQ, ncx;                                           // 16-byte complex elements
  size_t Op;                                                                              // 16-byte words (sliced)
  size_t Om0, Om1, Om2, Om3, X, V2, V3, Iv8, F, WB, Wc, Wd, Val, ExpT, ndbl;            // doubles
  size_t H0, H1, H2, H3, VH2, VL2, VH3, VL3, PM, nflt;                                     // floats
  size_t KLs, KLg, KLz, Sc, nint;                                                             // ints
  size_t Ent;                                                                             // uint16
  size_t Mult;                                                                            // bytes
  __host__ __device__ size_t bytes() const {
    return ncx * 16 + ndbl * 8 + nflt * 4 + nint * 4 + Ent * 2 + Mult + 16;
  }
};

__host__ __device__ inline PairCarve make_pair_carve(int nb, int J, int G, int nquart, int nT, int nS, int threads,
                                                   bool sliced) {
  PairCarve c;
  const size_t nb2 = (size_t)nb * nb, na = nb / 3, nwarps = ((size_t)threads + 31) / 32;
  size_t o = 0;
  c.E0 = o; o += (size_t)J * nb;
  c.E1 = o; o += nb2;
  c.E2 = o; o += sliced ? 0 : nb2;
  c.E3 = o; o += sliced ? 0 : nb2;
  c.Psi = o; o += (size_t)J * nb * G * 9;
  // T blocks (j0, x), padded by one entry; sliced: rows of digits of A and then of T, later |W|^2 and the lists
  c.T = o; o += sliced ? nwarps * 32 * (nb == 6 ? 36 : 76) / 4 : (size_t)J * nb * (nb2 + 1);
  c.Tw2 = o; o += G;
  // phases of the prologue; sliced: then the weak terms [S1, S4, S5][j0 x][largest of each sum, count]
  const size_t weak = sliced ? (3 * (size_t)J * nb * (nS + 1) + 3) / 4 : 0;
  c.TwQ = o; o += weak > (size_t)nquart ? weak : (size_t)nquart;
  c.Op = o; o += sliced ? 2 * 6 * (nb == 6 ? 2 * 32 * 2 : 3 * 32 * 3) / 4 : 0;
  c.ncx = o;
  size_t d = 0;
  c.Om0 = d; d += J;
  c.Om1 = d; d += nb;
  c.Om2 = d; d += nb;
  c.Om3 = d; d += nb;
  c.X = d; d += 2 * (size_t)J * nb;    // wa + wb, wa - wb  [j0][x]
  c.V2 = d; d += 3 * nb;
  c.V3 = d; d += 3 * nb;
  c.Iv8 = d; d += 2 * nb2;             // 8/sigma (or -1: delta := 1) of |v2 - v3| and |v2 + v3|, [y][j3]
  c.F = d; d += 3 * nb2;               // (1/sigma) x constants of P1, P2, P3 (x c and d weights for one temperature)
  c.WB = d; d += nS > 1 ? 3 * (size_t)nT * nb2 : 0;  // c and d weights of P1, P2, P3 per temperature
  c.Wc = d; d += 2 * (size_t)nT * nb;  // (1+n)/w and n/w of k2
  c.Wd = d; d += 2 * (size_t)nT * nb;  // and of k3
  c.Val = d; d += sliced ? 0 : nwarps * kPairCap;
  c.ExpT = d; d += kExpTab;
  c.ndbl = d;
  size_t f = 0;
  c.H0 = f; f += J;
  c.H1 = f; f += nb;
  c.H2 = f; f += nb;
  c.H3 = f; f += nb;
  c.VH2 = f; f += 3 * nb;
  c.VL2 = f; f += 3 * nb;
  c.VH3 = f; f += 3 * nb;
  c.VL3 = f; f += 3 * nb;
  f = (f + 1) & ~size_t(1);
  c.PM = f; f += 4 * nb2;  // [tab][y][j3] (P~, margin)
  c.nflt = f;
  size_t k = 0;
  c.KLs = k; k += na + 1;
  c.KLg = k; k += G;
  c.KLz = k; k += na * na;
  c.Sc = k; k += sliced ? (size_t)J * nb : 0;
  c.nint = k;
  c.Ent = sliced ? 0 : nwarps * kPairCap;
  c.Mult = (size_t)J + nb;
  return c;
}

// x + y or x - y (the sign flipped in the integer pipe)
__device__ __forceinline__ double add_signed(double x, double y, bool plus) {
  return __dadd_rn(x, __hiloint2double(__double2hiint(y) ^ (plus ? 0 : 0x80000000), __double2loint(y)));
}

// exp_neg64 (fp_rates_kernel.cuh) of v = x^2 with the range test and the rounding of v to k kept off the FP64 compare and
// convert instructions: x^2 + 1.5 2^52 holds k = rint(v) in its low bits; k - x^2 is rounded once
__device__ __forceinline__ double pair_exp_neg64(double x, const double* tab) {
  if ((__double2hiint(x) & 0x7fffffff) > 0x40300000) return exp(-(x * x) * kExpH);  // |x| >= 16 (1 + 2^-20) (also NaN)
  const double vm = fma(x, x, slices::kMagic);
  const int k = __double2loint(vm);
  const double t = fma(-x, x, __dsub_rn(vm, slices::kMagic));
  double p = (1.0 / 120.0) / 1073741824.0;
  p = fma(p, t, (1.0 / 24.0) / 16777216.0);
  p = fma(p, t, (1.0 / 6.0) / 262144.0);
  p = fma(p, t, 0.5 / 4096.0);
  p = fma(p, t, kExpH);
  p = fma(p, t, 1.0);
  return tab[k] * p;
}

// exp of the second order of {c, d} averaged in (rare: out of line)
__device__ __noinline__ double pair_two_orders(double ex, double z8, const double* tab) {
  return 0.5 * (ex + pair_exp_neg64(z8, tab));
}

// a weak term (rare: out of line): its number, and per sum the largest factor by its high word (shared memory adds doubles
// in a loop of compare and swap)
__device__ __noinline__ void pair_weak(int* wk, int nS, int lo, int nT, double gv, const double* wb, int stride) {
  atomicAdd(wk + nS, 1);
  for (int t = 0; t < nT; ++t) atomicMax(wk + lo + t, __double2hiint(wb ? gv * wb[t * stride] : gv));
}

// NB branches, up to MAXT sums per row.  DF: vertex contraction in double-float on the FP32 pipes (the terms in FP64: the
// weights of c and d fall as exp(-hbar (wc + wd) / k_B T), out of FP32's range at 10 to 20 K).  SL: both vertex contractions on the tensor cores in exact slices (fp_slices.cuh; unit eigenvectors, nb = 6 or 12): A in FP64,
// T as digits, |W|^2 of every entry in FP64.
template <int NB, int MAXT, bool DF, bool SL>
__global__ void __launch_bounds__(pair_threads_for(NB), pair_blocks_for(NB)) pair_kernel(RatesArgs a) {
  static_assert(!(DF && SL), "the double-float contraction has no sliced form");
  constexpr int NB2 = NB * NB, NA = NB / 3;
  using C = Cx<double>;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ long long s_item;
  __shared__ unsigned s_umask;
  __shared__ double s_up[kMaxT], s_down[kMaxT];  // scale of the c and d weights, and its inverse square
  const int J = a.J, G = a.G, nT = a.nT, nS = a.nS, N = a.N;  // nS sums per row: temperatures x parts
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const int rows = J * NB2;
  const PairCarve cv = make_pair_carve(NB, J, G, a.nquart, nT, a.nS, nthr, SL);
  C* cx = reinterpret_cast<C*>(smem);
  C *sE0 = cx + cv.E0, *sE1 = cx + cv.E1, *sE2 = cx + cv.E2, *sE3 = cx + cv.E3;
  C *sPsi = cx + cv.Psi, *sT = cx + cv.T, *sTw2 = cx + cv.Tw2, *sTwQ = cx + cv.TwQ;
  double* db = reinterpret_cast<double*>(cx + cv.ncx);
  double *sOm0 = db + cv.Om0, *sOm1 = db + cv.Om1, *sOm2 = db + cv.Om2, *sOm3 = db + cv.Om3;
  double *sV2 = db + cv.V2, *sV3 = db + cv.V3, *sWc = db + cv.Wc, *sWd = db + cv.Wd;
  double *sX = db + cv.X, *sIv8 = db + cv.Iv8, *sF = db + cv.F, *sWB = db + cv.WB, *sExpT = db + cv.ExpT;
  // sliced: W [j0 x][y][j3] (combine_magic) and the lists take the place of the digits once these are in registers
  double2* sW = reinterpret_cast<double2*>(sT);
  unsigned* sDig = reinterpret_cast<unsigned*>(sT);
  const unsigned* sOp = reinterpret_cast<const unsigned*>(cx + cv.Op);
  double* sVal = (SL ? reinterpret_cast<double*>(sW + (size_t)J * NB * NB2) : db + cv.Val) + (size_t)warp * kPairCap;
  double* sRed = reinterpret_cast<double*>(sT);  // the T block, free outside the k2 loop
  int* sWeak = reinterpret_cast<int*>(sTwQ);
  float* fb = reinterpret_cast<float*>(db + cv.ndbl);
  float *sH0 = fb + cv.H0, *sH1 = fb + cv.H1, *sH2 = fb + cv.H2, *sH3 = fb + cv.H3;
  float *sVH2 = fb + cv.VH2, *sVL2 = fb + cv.VL2, *sVH3 = fb + cv.VH3, *sVL3 = fb + cv.VL3;
  float2* sPM = reinterpret_cast<float2*>(fb + cv.PM);
  int* ib = reinterpret_cast<int*>(fb + cv.nflt);
  int *sKLs = ib + cv.KLs, *sKLg = ib + cv.KLg, *sKLz = ib + cv.KLz;
  int* sSc = ib + cv.Sc;
  unsigned short* sEnt = (SL ? reinterpret_cast<unsigned short*>(reinterpret_cast<double*>(sW + (size_t)J * NB * NB2) +
                                                                (size_t)((nthr + 31) / 32) * kPairCap)
                             : reinterpret_cast<unsigned short*>(ib + cv.nint)) + (size_t)warp * kPairCap;
  unsigned char* sMa = reinterpret_cast<unsigned char*>(reinterpret_cast<unsigned short*>(ib + cv.nint) + cv.Ent);
  unsigned char* sMb = sMa + J;

  const bool has_row = tid < rows;
  const int rjj = tid / NB2, rj1 = (tid / NB) % NB, rc = tid % NB;
  // complex elements of the block of T, free until Psi is complete
  const int kTabU = SL ? (nthr / 32) * 32 * (NB == 6 ? 36 : 76) / 4 : J * NB * (NB2 + 1);
  const size_t NM = (size_t)N * NB;
  const bool f32_sigma = a.dq_mode == 0;
  const double inv_sbdq = 1.0 / (a.sb * a.dq);
  const bool unit = a.unit_vertex != 0;
  // part of a test: by normal (0) and Umklapp (1), or by channel ++, +-, --
  auto part_of = [&](int kind, unsigned um) {
    return a.split == 0 ? 0 : a.split == 1 ? (int)((um >> kind) & 1u) : kind == 0 ? 1 : kind < 3 ? 0 : 2;
  };

  for (int o = tid; o < kExpTab; o += nthr) sExpT[o] = exp(-(double)o * kExpH);
  for (int t = tid; t < nT; t += nthr) {
    // at most 2^430: the largest sums, 2^860 times |W|^2 in units of 2^-102, stay below 2^1024
    const double half = 0.72134752044448170 * kHbar * a.wmax[0] / (kBoltzmann * a.T[t]);  // x / (2 ln 2)
    const int k = a.unit_weights && t == 0 ? 0 : __double2int_rn(fmin(half, 430.0));
    s_up[t] = scalbn(1.0, k);
    s_down[t] = scalbn(1.0, -2 * k);
  }
  for (int o = tid; o < NA + 1; o += nthr) sKLs[o] = a.pk_start[o];
  for (int o = tid; o < G; o += nthr) sKLg[o] = a.pk_grp[o];
  for (int o = tid; o < NA * NA; o += nthr) sKLz[o] = a.pk_zero[o];

  for (;;) {
    __syncthreads();  // the tables above; at later items, the last epilogue's reads
    if (tid == 0) s_item = (long long)atomicAdd(a.counter, 1ULL);
    __syncthreads();
    const long long item = s_item;
    if (item >= a.n_items) break;
    const int chunk = (int)(item % a.nchunk);
    const long long rest = item / a.nchunk;
    const int qi = (int)(rest % a.nq_sel);
    const int tile = (int)((rest / a.nq_sel) % a.ntile), seg = (int)(rest / a.nq_sel / a.ntile);
    const int q = a.qlist[qi];
    const int j0b = chunk * J;
    const int g[3] = {q / (a.grid[1] * a.grid[2]), (q / a.grid[2]) % a.grid[1], q % a.grid[2]};

    for (int o = tid; o < J * NB; o += nthr) sE0[o] = ld_e<double>(a, ((size_t)q * NB + j0b) * NB + o);
    for (int jj = tid; jj < J; jj += nthr) {
      const int m = q * NB + j0b + jj;
      const double w = a.omega[m];
      sOm0[jj] = w;
      sH0[jj] = a.omh[m];
      sMa[jj] = w > 0.0 ? a.mult[m] : 0;
    }
    double dir = 0.0;                  // tile mode: running direct sum of output tid
    unsigned long long dir_n = 0;
    unsigned cnt0 = 0, cnt1 = 0, cnt2 = 0, nwf = 0, nte = 0;
    unsigned long long niter = 0, npair = 0;

    const int k1_begin = tile * a.t1;
    const int k1_end = min(N, k1_begin + a.t1);
    const int k1_step = unit ? a.k1_stride : 1;
    const int k1_first = unit ? ((k1_begin + a.k1_stride - 1) / a.k1_stride) * a.k1_stride : k1_begin;
    for (int k1 = k1_first; k1 < k1_end; k1 += k1_step) {
      const PairRole role = pair_role(a, qi, q, k1);
      if (!role.run) continue;  // written by the mirrored pair
      const bool mir = role.mirror >= 0;
      const int rq = mir ? a.qlist[role.mirror] : 0;
      const int g1[3] = {k1 / (a.grid[1] * a.grid[2]), (k1 / a.grid[2]) % a.grid[1], k1 % a.grid[2]};
      __syncthreads();  // the previous pair's epilogue and, at the first pair, the tables of q
      for (int o = tid; o < NB2; o += nthr) sE1[o] = ld_e<double>(a, (size_t)k1 * NB2 + o);
      for (int o = tid; o < NB; o += nthr) {
        const double w = a.omega[k1 * NB + o];
        sOm1[o] = w;
        sH1[o] = a.omh[k1 * NB + o];
        sMb[o] = mir && w > 0.0 ? a.mult[rq * NB + o] : 0;
      }
      if (a.psi_u)
        for (int t = tid; t < a.nterm; t += nthr) {
          const int* m = a.term_meta + 4 * t;
          int e = 0;  // each term is below L, so e < 3 L
          for (int d = 0; d < 3; ++d) e += a.Lfac[d] * wrapi(g1[d] * m[1 + d], a.grid[d]);
          while (e >= a.L) e -= a.L;
          sTwQ[t] = ld_tw<double>(a, e);
        }
      for (int Q = tid; Q < (a.psi_u ? 0 : a.nquart); Q += nthr) {
        const int* m = a.qmeta + 9 * Q;
        int e = 0;  // each term is below L, so e < 3 L
        for (int d = 0; d < 3; ++d) e += a.Lfac[d] * wrapi(g1[d] * m[3 + d] - (g[d] + g1[d]) * m[6 + d], a.grid[d]);
        while (e >= a.L) e -= a.L;
        sTwQ[Q] = ld_tw<double>(a, e);
      }
      __syncthreads();
      int any = 0;
      for (int jj = 0; jj < J; ++jj) any |= sMa[jj];
      for (int x = 0; x < NB; ++x) any |= sMb[x];
      for (int o = tid; o < J * NB; o += nthr) {
        const int jj = o / NB, x = o % NB;
        sX[o] = __dadd_rn(sOm0[jj], sOm1[x]);
        sX[J * NB + o] = __dsub_rn(sOm0[jj], sOm1[x]);
      }
      // Psi[jj][j1][grp][gt] (see fp_rates_kernel.cuh): one thread per (jj, j1, grp) and block of three (gamma, theta)
      constexpr int kGtb = 3;
      if (a.psi_u && !unit && any) {
        // with U of this q at hand (psi_u_kernel): Psi = sum over the group's terms and beta of exp(i q'.(R_j - R_l)) e1_beta
        // U, 36 FMAs per term and three (gamma, theta) instead of 90 per quartet
        const double2* U = a.psi_u + ((size_t)qi * NB + j0b) * a.nterm * 27;
        // exp(i q'.(R_j - R_l)) e1 [j1][term][beta] where it fits into the block of T
        const bool table = 3 * NB * a.nterm <= kTabU;
        if (table) {
          for (int o = tid; o < 3 * NB * a.nterm; o += nthr) {
            const int t = (o / 3) % a.nterm;
            sT[o] = cmul(sTwQ[t], sE1[(o / (3 * a.nterm)) * NB + 3 * a.term_meta[4 * t] + o % 3]);
          }
          __syncthreads();
        }
        for (int o = tid; o < J * NB * G * (9 / kGtb); o += nthr) {
          const int gb = o % (9 / kGtb), jr = (o / (9 / kGtb)) % (J * NB), grp = o / ((9 / kGtb) * J * NB);
          const int j1 = jr % NB, jj = jr / NB;
          C sum[kGtb];
#pragma unroll
          for (int u = 0; u < kGtb; ++u) sum[u] = cmk<double>(0, 0);
          for (int t = a.term_start[grp]; t < a.term_start[grp + 1]; ++t) {
            const double2* uq = U + ((size_t)jj * a.nterm + t) * 27 + gb * kGtb;
            const C* e1 = table ? sT + 3 * ((size_t)j1 * a.nterm + t) : sE1 + j1 * NB + 3 * a.term_meta[4 * t];
#pragma unroll
            for (int be = 0; be < 3; ++be) {
              const C et = table ? e1[be] : cmul(sTwQ[t], e1[be]);
#pragma unroll
              for (int u = 0; u < kGtb; ++u) {
                const double2 v = uq[be * 9 + u];
                cfma(sum[u], et, cmk<double>(v.x, v.y));
              }
            }
          }
#pragma unroll
          for (int u = 0; u < kGtb; ++u) {
            const size_t at = (size_t)(jr * G + grp) * 9 + gb * kGtb + u;
            if constexpr (DF)
              reinterpret_cast<float4*>(sPsi)[at] = cdf_from(sum[u].re, sum[u].im);
            else
              sPsi[at] = sum[u];
          }
        }
      }
      const int npsi = a.psi_u || unit || !any ? 0 : J * NB * G * (9 / kGtb);
      for (int o = tid; o < npsi; o += nthr) {
        const int gb = o % (9 / kGtb);
        const int jr = (o / (9 / kGtb)) % (J * NB);
        const int grp = o / ((9 / kGtb) * J * NB);
        const int t9 = jr * G + grp;
        const int j1 = jr % NB, jj = jr / NB;
        C sum[kGtb];
#pragma unroll
        for (int u = 0; u < kGtb; ++u) sum[u] = cmk<double>(0, 0);
        for (int qq = a.grp_qstart[grp]; qq < a.grp_qstart[grp + 1]; ++qq) {
          const int Q = a.grp_q[qq];
          const int ia = a.qmeta[9 * Q], ja = a.qmeta[9 * Q + 1];
          C p[9];
#pragma unroll
          for (int al = 0; al < 3; ++al) {
            const C e0 = sE0[jj * NB + 3 * ia + al];
#pragma unroll
            for (int be = 0; be < 3; ++be) p[al * 3 + be] = cmul(e0, sE1[j1 * NB + 3 * ja + be]);
          }
          const C tq = sTwQ[Q];
          const size_t fo = 81 * (size_t)Q + gb * kGtb;
#pragma unroll
          for (int u = 0; u < kGtb; ++u) {
            C s = cmk<double>(0, 0);
#pragma unroll
            for (int ab = 0; ab < 9; ++ab) {
              const double fv = a.qfc[fo + ab * 9 + u];
              s.re = fma(fv, p[ab].re, s.re);
              s.im = fma(fv, p[ab].im, s.im);
            }
            cfma(sum[u], tq, s);
          }
        }
#pragma unroll
        for (int u = 0; u < kGtb; ++u) {
          if constexpr (DF)
            reinterpret_cast<float4*>(sPsi)[(size_t)t9 * 9 + gb * kGtb + u] = cdf_from(sum[u].re, sum[u].im);
          else
            sPsi[(size_t)t9 * 9 + gb * kGtb + u] = sum[u];
        }
      }

      if constexpr (SL) {
        // scale of every (j0, x): 2^s above the Frobenius norm of its A block for any phases, so above every element of
        // A, T and W (unit eigenvectors)
        double* sB = reinterpret_cast<double*>(sT);
        __syncthreads();
        for (int o = tid; o < 3 * J * NB * (nS + 1); o += nthr) sWeak[o] = 0;
        if (!unit && any) {
          for (int o = tid; o < J * NB * NB2; o += nthr) {
            const int ab = o / NB2, k = (o / NB) % NB, l = o % NB;
            const C* ps = sPsi + (size_t)ab * G * 9 + (k % 3) * 3 + l % 3;
            double sum = 0.0;
            auto take = [&](int grp) {  // |z| <= max + (sqrt 2 - 1) min
              const C z = ps[grp * 9];
              const double u = fabs(z.re), v = fabs(z.im);
              sum += fmax(u, v) + 0.41421357 * fmin(u, v);
            };
            if (sKLz[(k / 3) * NA + l / 3] >= 0) take(sKLz[(k / 3) * NA + l / 3]);
            for (int gi = sKLs[k / 3]; gi < sKLs[k / 3 + 1]; ++gi)
              if (sKLg[gi] >> 24 == l / 3) take(sKLg[gi] & 0xffffff);
            sB[o] = sum * sum;
          }
          __syncthreads();
          for (int ab = tid; ab < J * NB; ab += nthr) {
            double f = 0.0;
            for (int o = 0; o < NB2; ++o) f += sB[ab * NB2 + o];
            sSc[ab] = f > 0.0 ? (f < 1e300 ? ilogb(sqrt(f) * 1.0001) + 1 : 1000) : -600;  // -600: W is zero, not weak
          }
        }
      }

      const unsigned ma = has_row ? sMa[rjj] : 0u, mb = has_row ? sMb[rj1] : 0u;
      const bool active = (ma | mb) != 0;
      // candidates of this row: P1, P2, P3 while either mode is wanted, P4 for a, P5 for b
      const unsigned row_cand = (active ? 7u : 0u) | (ma ? 8u : 0u) | (mb ? 16u : 0u);
      // process_mask as P1 = bit 1 (+-), P2 = P3 = bit 0 (++), P4 = P5 = bit 2 (--)
      const unsigned proc_cand = ((a.cand_mask & 2u) ? 1u : 0u) | ((a.cand_mask & 1u) ? 6u : 0u) |
                                 ((a.cand_mask & 4u) ? 24u : 0u);
      // S1, S4 and S5 of the row; S1 in registers, the others (rarer) in local memory when there are several
      // temperatures
      double S1[MAXT], R45[2 * MAXT];
      unsigned n1 = 0, n4 = 0, n5 = 0;  // accepted terms of this pair: of both modes, of a only, of b only
#pragma unroll
      for (int t = 0; t < MAXT; ++t) S1[t] = 0.0;
      if constexpr (MAXT == 1) {
        R45[0] = R45[1] = 0.0;
      } else {
        for (int t = 0; t < 2 * nS; ++t) R45[t] = 0.0;
      }
      // value v of test `kind` at the entry e = (y, j3) into the row's sums, those of its part from slot lo
      unsigned umask = 0;  // Umklapp tests of the current k2
      auto add = [&](const double v, const int kind, const int e) {
        if constexpr (MAXT == 1) {
          if (kind < 3)
            S1[0] += v;
          else if (kind == 3)
            R45[0] += v;
          else
            R45[1] += v;
        } else {
          const double* wb = sWB + (kind < 3 ? kind : 0) * NB2 + e;
          const int lo = part_of(kind, umask) * nT;
          if (kind < 3) {
#pragma unroll
            for (int t = 0; t < MAXT; ++t) {
              if (t >= nS) break;
              if (t >= lo && t < lo + nT) S1[t] = fma(v, wb[3 * (t - lo) * NB2], S1[t]);
            }
          } else {
#pragma unroll 1
            for (int t = 0; t < nT; ++t) {
              double& r = R45[(kind - 3) * nS + lo + t];
              r = fma(v, wb[3 * t * NB2], r);
            }
          }
        }
      };
      __syncthreads();

      int g2[3] = {0, 0, 0};
      const int gs[3] = {(g[0] + g1[0]) % a.grid[0], (g[1] + g1[1]) % a.grid[1], (g[2] + g1[2]) % a.grid[2]};
      unsigned it = 0;
      int turn = seg;  // visits until the segment's next one
      for (int k2 = 0; any && k2 < N; ++k2) {
        if (k2 != 0 && ++g2[2] == a.grid[2]) {
          g2[2] = 0;
          if (++g2[1] == a.grid[1]) {
            g2[1] = 0;
            ++g2[0];
          }
        }
        int g3[3], gd[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          g3[d] = gs[d] + g2[d];
          if (g3[d] >= a.grid[d]) g3[d] -= a.grid[d];
          gd[d] = g3[d] ? a.grid[d] - g3[d] : 0;
        }
        const int k3 = (g3[0] * a.grid[1] + g3[1]) * a.grid[2] + g3[2];
        const int kd = (gd[0] * a.grid[1] + gd[1]) * a.grid[2] + gd[2];
        if (kd < k2) continue;  // {c, d} is visited at its smaller index
        if (turn-- != 0) continue;
        turn = a.nseg - 1;
        const bool twice = kd != k2;  // both orders of {c, d} come from this visit
        // ---- tables of k2 and k3
        if ((a.nu_select != 0 || a.split == 1) && tid == 0) s_umask = pair_umklapp_bits(a, g, g1, g2, g3);
        if constexpr (SL) {
          constexpr int kOp4 = slices::Shape<SL ? NB : 6>::kOperand / 4;
          const uint4* src = reinterpret_cast<const uint4*>(a.operands);
          uint4* dst = reinterpret_cast<uint4*>(cx + cv.Op);
          if (!unit)
            for (int o = tid; o < 2 * kOp4; o += nthr)
              dst[o] = src[(size_t)(o < kOp4 ? k3 : k2) * 2 * kOp4 + o];
        } else
        for (int o = tid; o < NB2; o += nthr) {
          const double2 e2v = a.evec[(size_t)k2 * NB2 + o], e3v = a.evec[(size_t)k3 * NB2 + o];
          if constexpr (DF) {
            reinterpret_cast<float4*>(sE2)[o] = cdf_from(e2v.x, e2v.y);
            reinterpret_cast<float4*>(sE3)[o] = cdf_from(e3v.x, e3v.y);
          } else {
            sE2[o] = cmk<double>(e2v.x, e2v.y);
            sE3[o] = cmk<double>(e3v.x, e3v.y);
          }
        }
        for (int o = tid; o < NB; o += nthr) {
          sOm2[o] = a.omega[k2 * NB + o];
          sOm3[o] = a.omega[k3 * NB + o];
          sH2[o] = a.omh[k2 * NB + o];
          sH3[o] = a.omh[k3 * NB + o];
        }
        for (int o = tid; o < 3 * NB; o += nthr) {
          sV2[o] = a.vel[(size_t)k2 * NB * 3 + o];
          sV3[o] = a.vel[(size_t)k3 * NB * 3 + o];
          sVH2[o] = a.velh[(size_t)k2 * NB * 3 + o];
          sVL2[o] = a.vell[(size_t)k2 * NB * 3 + o];
          sVH3[o] = a.velh[(size_t)k3 * NB * 3 + o];
          sVL3[o] = a.vell[(size_t)k3 * NB * 3 + o];
        }
        for (int o = tid; o < 2 * nT * NB; o += nthr) {
          const int t = o / (2 * NB), r = o % (2 * NB);
          const size_t base = 3 * ((size_t)t * NM);
          sWc[o] = a.wt[base + 3 * ((size_t)k2 * NB + r / 2) + 1 + r % 2] * s_up[t];
          sWd[o] = a.wt[base + 3 * ((size_t)k3 * NB + r / 2) + 1 + r % 2] * s_up[t];
        }
        for (int gi = tid; gi < G; gi += nthr) {
          const int* gm = a.gmeta + 5 * gi;
          int e = 0;
          for (int d = 0; d < 3; ++d) e += a.Lfac[d] * wrapi(g2[d] * gm[2 + d], a.grid[d]);
          while (e >= a.L) e -= a.L;
          if constexpr (DF) {
            const double2 t = a.tw[e];
            reinterpret_cast<float4*>(sTw2)[gi] = cdf_from(t.x, t.y);
          } else {
            sTw2[gi] = ld_tw<double>(a, e);
          }
        }
        __syncthreads();
        // ---- sigma tables and factors per (y, j3); A row and T row
        for (int o = tid; o < 2 * NB2; o += nthr) {
          const int tab = o / NB2, e = o % NB2, y = e / NB, j3 = e % NB;
          const double sgn = tab ? -1.0 : 1.0;
          double iv = -1.0;
          if (f32_sigma) {
            float inv;
            sigma_entry_f32(a, sVH2 + 3 * y, sVL2 + 3 * y, (float)sgn, sVH3 + 3 * j3, sVL3 + 3 * j3, sV2 + 3 * y,
                            sV3 + 3 * j3, sPM + o, &inv);
            // the Gaussian takes 1/sigma to a few ulp (CUDA's rsqrt); delta := 1 is the prefilter's exact decision
            if (inv >= 0.f) {
              const unsigned long long flip = tab ? 0x8000000000000000ULL : 0ULL;
              const double dx = __dsub_rn(__longlong_as_double(__double_as_longlong(sV2[3 * y]) ^ flip), sV3[3 * j3]);
              const double dy = __dsub_rn(__longlong_as_double(__double_as_longlong(sV2[3 * y + 1]) ^ flip), sV3[3 * j3 + 1]);
              const double dz = __dsub_rn(__longlong_as_double(__double_as_longlong(sV2[3 * y + 2]) ^ flip), sV3[3 * j3 + 2]);
              iv = rsqrt(fma(dx, dx, fma(dy, dy, dz * dz))) * inv_sbdq;
            }
          } else {
            double ex[2];
            float inv;
            sigma_entry(a, sV2 + 3 * y, sgn, sV3 + 3 * j3, ex);
            sigma_f_from_exact(ex, sPM + o, &inv);
            iv = ex[1];
          }
          sIv8[o] = iv >= 0.0 ? 8.0 * iv : -1.0;
          // 1/2 per order of {c, d} (Eq. tao0; the 1/6 of -- is completed in the epilogue) and the Gaussian's 1/sqrt(pi)
          const double f = iv >= 0.0 ? iv * kInvSqrtPi : 1.0;
          if (tab) {
            sF[e] = (twice ? 1.0 : 0.5) * f * (MAXT == 1 ? sWc[2 * y + 1] * sWd[2 * j3 + 1] : 1.0);
          } else {
            sF[NB2 + e] = 0.5 * f * (MAXT == 1 ? sWc[2 * y] * sWd[2 * j3 + 1] : 1.0);
            sF[2 * NB2 + e] = 0.5 * f * (MAXT == 1 ? sWc[2 * y + 1] * sWd[2 * j3] : 1.0);
          }
        }
        if constexpr (MAXT > 1)
          for (int o = tid; o < 3 * nT * NB2; o += nthr) {
            const int t = o / (3 * NB2), k = (o / NB2) % 3, y = (o / NB) % NB, j3 = o % NB;
            sWB[o] = sWc[2 * (t * NB + y) + (k == 1 ? 0 : 1)] * sWd[2 * (t * NB + j3) + (k == 2 ? 0 : 1)];
          }
        if (has_row && !unit) {
          const int ka = rc / 3, ga = rc % 3;
          const int g_begin = sKLs[ka], g_end = sKLs[ka + 1];
          if constexpr (DF) {
            float4 Ad[NB];
            const float4* psi_row = reinterpret_cast<const float4*>(sPsi) + (size_t)(rjj * NB + rj1) * G * 9 + ga * 3;
            const float4* twd = reinterpret_cast<const float4*>(sTw2);
#pragma unroll
            for (int l = 0; l < NA; ++l) {
              const int z = sKLz[ka * NA + l];
#pragma unroll
              for (int th = 0; th < 3; ++th)
                Ad[3 * l + th] = z >= 0 ? psi_row[z * 9 + th] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            float4 cur[3];
            int la = -1;
            auto put = [&]() {
#pragma unroll
              for (int l = 0; l < NA; ++l)
                if (l == la)
#pragma unroll
                  for (int th = 0; th < 3; ++th) Ad[3 * l + th] = cur[th];
            };
            for (int gi = g_begin; gi < g_end; ++gi) {
              const int code = sKLg[gi], grp = code & 0xffffff, lg = code >> 24;
              if (lg != la) {
                put();
                la = lg;
#pragma unroll
                for (int l = 0; l < NA; ++l)
                  if (l == la)
#pragma unroll
                    for (int th = 0; th < 3; ++th) cur[th] = Ad[3 * l + th];
              }
              const float4 tw = twd[grp];
              const float4* ps = psi_row + grp * 9;
#pragma unroll
              for (int th = 0; th < 3; ++th) cdf_mac(cur[th], tw, ps[th]);
            }
            put();
            const float4* e3d = reinterpret_cast<const float4*>(sE3);
            float4* trow = reinterpret_cast<float4*>(sT + (size_t)(rjj * NB + rj1) * (NB2 + 1) + rc * NB);
#pragma unroll
            for (int j3 = 0; j3 < NB; ++j3) {
              float4 sd = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
              for (int d = 0; d < NB; ++d) cdf_mac_conj(sd, Ad[d], e3d[j3 * NB + d]);
              trow[j3] = cdf_norm(sd);
            }
          } else {
            C Arow[NB];
            const C* psi_row = sPsi + (size_t)(rjj * NB + rj1) * G * 9 + ga * 3;
            // groups with D = 0 have the phase 1: they start the sums (no arithmetic)
#pragma unroll
            for (int l = 0; l < NA; ++l) {
              const int z = sKLz[ka * NA + l];
#pragma unroll
              for (int th = 0; th < 3; ++th) Arow[3 * l + th] = z >= 0 ? psi_row[z * 9 + th] : cmk<double>(0, 0);
            }
            // the other groups of atom ka in l order: lanes of different ka run about the same count
            C cur[3];
            int la = -1;
            auto put = [&]() {
#pragma unroll
              for (int l = 0; l < NA; ++l)
                if (l == la)
#pragma unroll
                  for (int th = 0; th < 3; ++th) Arow[3 * l + th] = cur[th];
            };
            for (int gi = g_begin; gi < g_end; ++gi) {
              const int code = sKLg[gi], grp = code & 0xffffff, lg = code >> 24;
              if (lg != la) {
                put();
                la = lg;
#pragma unroll
                for (int l = 0; l < NA; ++l)
                  if (l == la)
#pragma unroll
                    for (int th = 0; th < 3; ++th) cur[th] = Arow[3 * l + th];
              }
              const C tw = sTw2[grp];
              const C* ps = psi_row + grp * 9;
#pragma unroll
              for (int th = 0; th < 3; ++th) cfma(cur[th], tw, ps[th]);
            }
            put();
            if constexpr (SL) {
              const int sc = sSc[rjj * NB + rj1];
              unsigned* drow = sDig + tid * slices::Shape<SL ? NB : 6>::kRow;
#pragma unroll
              for (int d = 0; d < NB; ++d) {
                const unsigned long long vr = slices::fixed_from(Arow[d].re, sc), vi = slices::fixed_from(Arow[d].im, sc);
#pragma unroll
                for (int i = 0; i < slices::kDigits; ++i) drow[i * NB + d] = slices::pack_digit(i, vr, vi);
              }
            } else {
              C* trow = sT + (size_t)(rjj * NB + rj1) * (NB2 + 1) + rc * NB;
#pragma unroll
              for (int j3 = 0; j3 < NB; ++j3) {
                C s = cmk<double>(0, 0);
#pragma unroll
                for (int d = 0; d < NB; ++d) cfma_conj(s, Arow[d], sE3[j3 * NB + d]);
                trow[j3] = s;
              }
            }
          }
        }
        if constexpr (SL) {
          if (!unit) {
            // T = A conj(e3) and W = T e2 in slices; a warp's 32 rows are two row tiles.  Rows of A are (j0, x, k gamma);
            // the digits of T go to rows (j0, x, j3), which other warps may hold, so its fragments and stores are
            // separated by barriers
            using Sh = slices::Shape<SL ? NB : 6>;
            const int g = lane >> 2, t = lane & 3;
            unsigned af[2][slices::kDigits][Sh::kA];
            __syncwarp();
            slices::load_a<SL ? NB : 6>(sDig, warp * 32, lane, af[0]);
            slices::load_a<SL ? NB : 6>(sDig, warp * 32 + 16, lane, af[1]);
            __syncthreads();
#pragma unroll
            for (int nt = 0; nt < Sh::kTiles; ++nt) {
              unsigned bf[slices::kDigits][Sh::kB];
              slices::load_b<SL ? NB : 6>(sOp, nt, lane, bf);
#pragma unroll
              for (int mt = 0; mt < 2; ++mt) {
                float acc[slices::kLevels][4];
                slices::contract<SL ? NB : 6>(acc, af[mt], bf);
                float D[4][slices::kLevels];
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                  for (int s = 0; s < slices::kLevels; ++s) D[c][s] = acc[s][c];
                const int r0 = warp * 32 + mt * 16 + g;
                if (NB == 6 && nt == 1) {  // one real of branches 4, 5 per lane, of two rows
                  const unsigned long long v0 = slices::combine_fixed<NB>(D[0]), v1 = slices::combine_fixed<NB>(D[2]);
                  const int j = 4 + (t >> 1), ri = t & 1;
                  unsigned short* d0 = reinterpret_cast<unsigned short*>(sDig + ((r0 / NB) * NB + j) * Sh::kRow + r0 % NB) + ri;
                  unsigned short* d1 = reinterpret_cast<unsigned short*>(sDig + (((r0 + 8) / NB) * NB + j) * Sh::kRow + (r0 + 8) % NB) + ri;
#pragma unroll
                  for (int i = 0; i < slices::kDigits; ++i) {
                    const unsigned w = slices::pack_digit(i, v0, v1);
                    if (r0 < rows) d0[2 * i * NB] = (unsigned short)w;
                    if (r0 + 8 < rows) d1[2 * i * NB] = (unsigned short)(w >> 16);
                  }
                } else {
#pragma unroll
                  for (int h = 0; h < 2; ++h) {
                    const int r = r0 + 8 * h;
                    const unsigned long long vr = slices::combine_fixed<NB>(D[2 * h]), vi = slices::combine_fixed<NB>(D[2 * h + 1]);
                    unsigned* drow = sDig + ((r / NB) * NB + nt * 4 + t) * Sh::kRow + r % NB;
                    if (r < rows)
#pragma unroll
                      for (int i = 0; i < slices::kDigits; ++i) drow[i * NB] = slices::pack_digit(i, vr, vi);
                  }
                }
              }
            }
            __syncthreads();
            slices::load_a<SL ? NB : 6>(sDig, warp * 32, lane, af[0]);
            slices::load_a<SL ? NB : 6>(sDig, warp * 32 + 16, lane, af[1]);
            __syncthreads();
#pragma unroll
            for (int nt = 0; nt < Sh::kTiles; ++nt) {
              unsigned bf[slices::kDigits][Sh::kB];
              slices::load_b<SL ? NB : 6>(sOp + Sh::kOperand, nt, lane, bf);
#pragma unroll
              for (int mt = 0; mt < 2; ++mt) {
                float acc[slices::kLevels][4];
                slices::contract<SL ? NB : 6>(acc, af[mt], bf);
                float D[4][slices::kLevels];
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                  for (int s = 0; s < slices::kLevels; ++s) D[c][s] = acc[s][c];
                const int r0 = warp * 32 + mt * 16 + g;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                  const int r = r0 + 8 * h, at = (r / NB) * NB2 + r % NB;  // row (j0, x, j3): entry [j0 x][y][j3]
                  const double x = slices::combine_magic<NB>(D[2 * h]);
                  if (NB == 6 && nt == 1) {
                    if (r < rows) reinterpret_cast<double*>(sW + at + (4 + (t >> 1)) * NB)[t & 1] = x;
                  } else {
                    const double y = slices::combine_magic<NB>(D[2 * h + 1]);
                    if (r < rows) sW[at + (nt * 4 + t) * NB] = make_double2(x, y);
                  }
                }
              }
            }
            if (has_row) nwf += NB;
          }
        }
        __syncthreads();
        // ---- window tests of the row's entries and evaluation of the accepted ones
        {
          if (a.split == 1) umask = s_umask;
          const int x = rj1, y = rc, jq = has_row ? rjj : 0;
          const unsigned cand = row_cand & proc_cand &
                                (a.nu_select == 0 ? 31u : a.nu_select == 1 ? ~s_umask : s_umask) &
                                (twice ? 31u : ~4u);  // c = d: P3 at (y, j3) is P2 at (j3, y)
          const float h0 = sH0[jq], hx = sH1[x], hy = sH2[y];
          const bool row_ok = active && h0 != 0.f && hx != 0.f && hy != 0.f;
          const float hab = h0 + hx, dab = h0 - hx, sab = hab + hy;
          const unsigned wsum = ma + mb, o1 = twice ? 2u : 1u;
#pragma unroll 1
          for (int jb = 0; jb < NB; jb += kPairGroup) {
            constexpr int kG = NB < kPairGroup ? NB : kPairGroup;
            // accepted (test, j3): bit kind * kPairGroup + u; `lone`: only one of the test's two orders is accepted
            unsigned m = 0, lone = 0;
            if (row_ok) {
#pragma unroll
              for (int u = 0; u < kG; ++u) {
                const int j3 = jb + u;
                const float h3 = sH3[j3];
                if (h3 == 0.f) continue;
                const float sS = kRelS * (sab + h3);
                const float hs = hy + h3, hd = hy - h3;
                const float2 p0 = sPM[y * NB + j3], p1 = sPM[NB2 + y * NB + j3];
                // settled by more than the prefilter's rounding, or in the band that the FP64 definition decides
                unsigned acc = 0, band = 0;
                auto test = [&](int kind, float d, float P, float M) {
                  acc |= (d < P - M ? 1u : 0u) << kind;
                  band |= (d <= P + M && !(d < P - M) ? 1u : 0u) << kind;
                };
                const float M0 = sS + p0.y, M1 = sS + p1.y;
                test(0, fabsf(hab - hs), p1.x, M1);
                // P2 and P3 (P4 and P5) share the smaller |dw~|: | hab - |hy - h3| | (| hs - |h0 - hx| |)
                if (fabsf(hab - fabsf(hd)) <= p0.x + M0) {
                  test(1, fabsf(hab + hd), p0.x, M0);
                  test(2, fabsf(hab - hd), p0.x, M0);
                }
                if (fabsf(hs - fabsf(dab)) <= p1.x + M1) {
                  test(3, fabsf(dab - hs), p1.x, M1);
                  test(4, fabsf(dab + hs), p1.x, M1);
                }
                acc &= cand;
                band &= cand;
                while (band) {
                  const int kind = __ffs(band) - 1;
                  band &= band - 1;
                  // FP64 decisions in the operation order of the definition, for each order of {c, d}
                  const double w0 = sOm0[jq], w1 = sOm1[x], w2 = sOm2[y], w3 = sOm3[j3];
                  const bool tab1 = kind != 1 && kind != 2;
                  double ex[2];
                  sigma_entry(a, sV2 + 3 * y, tab1 ? -1.0 : 1.0, sV3 + 3 * j3, ex);
                  const double s = kind < 3 ? __dadd_rn(w0, w1) : kind == 3 ? __dsub_rn(w0, w1) : __dsub_rn(w1, w0);
                  const double d1 = kind == 1   ? __dsub_rn(__dadd_rn(s, w2), w3)
                                    : kind == 2 ? __dsub_rn(__dadd_rn(s, w3), w2)
                                                : __dsub_rn(__dsub_rn(s, w2), w3);
                  const bool in1 = fabs(d1) <= ex[0];
                  const bool in2 = tab1 && twice ? fabs(__dsub_rn(__dsub_rn(s, w3), w2)) <= ex[0] : in1;
                  if (in1 || in2) acc |= 1u << kind;
                  if (in1 != in2) lone |= 1u << (kind * kPairGroup + u);
                }
#pragma unroll
                for (int kind = 0; kind < 5; ++kind) m |= ((acc >> kind) & 1u) << (kind * kPairGroup + u);
              }
              constexpr unsigned kM = (1u << kPairGroup) - 1u;
              const unsigned c1 = o1 * __popc(m & kM) - __popc(lone & kM);
              const unsigned c23 = __popc(m & (kM << kPairGroup | kM << (2 * kPairGroup)));
              const unsigned c4 = o1 * __popc(m & (kM << (3 * kPairGroup))) - __popc(lone & (kM << (3 * kPairGroup)));
              const unsigned c5 = o1 * __popc(m & (kM << (4 * kPairGroup))) - __popc(lone & (kM << (4 * kPairGroup)));
              cnt0 += wsum * c23;
              cnt1 += wsum * c1;
              cnt2 += ma * c4 + mb * c5;
              n1 += c1 + c23;
              n4 += c4;
              n5 += c5;
            }
            // compacted in lane order, test by test within a lane
            const int nmy = __popc(m);
            nte += nmy;
            if (!SL && !unit) nwf += nmy;
            int incl = nmy;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const int v = __shfl_up_sync(0xffffffffu, incl, o);
              if (lane >= o) incl += v;
            }
            const int total = __shfl_sync(0xffffffffu, incl, 31);
            int pos = incl - nmy;
            unsigned left = m;
            for (int r0 = 0; r0 < total; r0 += kPairCap) {
              const int rn = min(total - r0, kPairCap);
              const int pos0 = pos;
              const unsigned left0 = left;
              for (; left && pos < r0 + kPairCap; left &= left - 1) {
                const int bit = __ffs(left) - 1;
                sEnt[pos++ - r0] = (unsigned short)(lane | bit << 5 | ((lone >> bit) & 1u) << 10);
              }
              __syncwarp();
              for (int i = lane; i < rn; i += 32) {
                const unsigned en = sEnt[i];
                const int row = (tid & ~31) + (int)(en & 31u), bit = (int)(en >> 5) & 31;
                const int kind = bit / kPairGroup, j3 = jb + bit % kPairGroup;
                const int ejj = row / NB2, ex = (row / NB) % NB, ey = row % NB;
                const int ab = ejj * NB + ex, e = ey * NB + j3;
                const bool tab0 = kind == 1 || kind == 2;
                const double iv8 = sIv8[(tab0 ? 0 : NB2) + e];
                double gv = sF[(tab0 ? kind : 0) * NB2 + e];
                // dw in the operation order of the definition (P5 negated): at a resonance of a mode with itself it is
                // a rounding error, which a small sigma makes visible
                const double wx = sX[(kind >= 3 ? J * NB : 0) + ab];
                const double wc = sOm2[ey], wd = sOm3[j3];
                const double y1 = kind == 2 ? wd : wc, y2 = kind == 2 ? wc : wd;
                const bool plus1 = kind == 1 || kind == 2 || kind == 4, plus2 = kind == 4;
                const double dw = add_signed(add_signed(wx, y1, plus1), y2, plus2);
                // the other order of {c, d} differs by its rounding, which only a sigma below 1e-3 rad/ps shows
                const bool orders = twice && !tab0 && !(en & 1024u);
                double W2 = 1.0;
                if constexpr (DF) {
                  if (!unit) {
                    const float4* tb = reinterpret_cast<const float4*>(sT + (size_t)ab * (NB2 + 1) + j3);
                    const float4* e2 = reinterpret_cast<const float4*>(sE2 + ey * NB);
                    float4 Wd = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int c = 0; c < NB; ++c) cdf_mac(Wd, e2[c], tb[c * NB]);
                    W2 = cdf_abs2(cdf_norm(Wd));  // a vanishing W leaves its high parts cancelled
                  }
                } else if constexpr (SL) {
                  if (!unit) {
                    const double2 w = sW[ab * NB2 + e];
                    const double wr = w.x - slices::kMagic, wi = w.y - slices::kMagic;
                    W2 = fma(wr, wr, wi * wi);
                  }
                } else if (!unit) {
                  const C* tb = sT + (size_t)ab * (NB2 + 1) + j3;
                  const C* e2 = sE2 + ey * NB;
                  C Wv = cmk<double>(0, 0);
#pragma unroll
                  for (int c = 0; c < NB; ++c) cfma(Wv, e2[c], tb[c * NB]);
                  W2 = Wv.re * Wv.re + Wv.im * Wv.im;
                }
                if (__double2hiint(iv8) >= 0) {  // not -1 (delta := 1)
                  const double x8 = dw * iv8;
                  double ex = pair_exp_neg64(x8, sExpT);
                  if (__double2hiint(iv8) > 0x40bf4000 && orders)  // 8 / sigma > 8000
                    ex = pair_two_orders(ex, add_signed(add_signed(wx, y2, plus1), y1, plus2) * iv8, sExpT);
                  gv *= ex;
                }
                if (en & 1024u) gv *= 0.5;
                const double v = W2 * gv;
                if constexpr (SL) {
                  // |W|^2 is in units of (2^(s - 51))^2
                  if (__double2hiint(W2) < (1023 + 102 + 2 * slices::kWeakExponent) << 20 && !unit) {
                    pair_weak(sWeak + ((kind < 3 ? 0 : kind - 2) * J * NB + ab) * (nS + 1), nS,
                              MAXT == 1 ? 0 : part_of(kind, umask) * nT, MAXT == 1 ? 1 : nT, gv,
                              MAXT == 1 ? nullptr : sWB + (kind < 3 ? kind : 0) * NB2 + e, 3 * NB2);
                  }
                }
                sVal[i] = v;
              }
              __syncwarp();
              int p = pos0 - r0;
              // the three sums one after the other: a warp runs the longest list of each, not all three per position
              const unsigned done = left0 & ~left;
              constexpr unsigned kM = (1u << kPairGroup) - 1u;
              for (unsigned b = done & ((1u << (3 * kPairGroup)) - 1u); b; b &= b - 1) {
                const int bit = __ffs(b) - 1;
                add(sVal[p++], bit / kPairGroup, y * NB + jb + bit % kPairGroup);
              }
              for (unsigned b = done >> (3 * kPairGroup) & kM; b; b &= b - 1) add(sVal[p++], 3, y * NB + jb + __ffs(b) - 1);
              for (unsigned b = done >> (4 * kPairGroup) & kM; b; b &= b - 1) add(sVal[p++], 4, y * NB + jb + __ffs(b) - 1);
              __syncwarp();
            }
          }
        }
        ++it;
        __syncthreads();
      }
      niter += it;
      npair += any ? 1 : 0;
      // ---- R(a; b) of the chunk's j0 and R(b; a) of every x, rows summed in a fixed order
      const size_t first = (size_t)seg * a.nq_sel * N * a.nchunk;  // slots of the segment
      const size_t slot = a.mirror ? first + ((size_t)qi * N + k1) * a.nchunk + chunk : 0;
      const size_t mslot = mir ? first + ((size_t)role.mirror * N + role.mirror_b) * a.nchunk + chunk : 0;
      const int nout = J + (mir ? NB : 0);
      for (int t = 0; t < nS; ++t) {
        if (has_row) {
          double s1 = 0.0;
#pragma unroll
          for (int tt = 0; tt < MAXT; ++tt)
            if (tt == t) s1 = S1[tt];
          // sliced: |W|^2 was in units of (2^(s - 51))^2
          const double f = SL && !unit && any ? scalbn(1.0, 2 * sSc[rjj * NB + rj1] - 102) : 1.0;
          sRed[tid] = f * s1;
          sRed[rows + tid] = f * R45[t];
          sRed[2 * rows + tid] = f * R45[nS + t];
        }
        __syncthreads();
        if (tid < nout) {
          const bool direct = tid < J;
          const int m = direct ? tid : tid - J;
          const double* W = a.wt + 3 * (size_t)(t % nT) * NM;
          double sum = 0.0;
          for (int o = 0; o < (direct ? NB : J); ++o) {
            const int r0 = ((direct ? m : o) * NB + (direct ? o : m)) * NB;
            double s1 = 0.0, s2 = 0.0;
            for (int yy = 0; yy < NB; ++yy) {
              s1 += sRed[r0 + yy];
              s2 += sRed[(direct ? rows : 2 * rows) + r0 + yy];
            }
            const double* wo = W + 3 * (direct ? (size_t)k1 * NB + o : (size_t)q * NB + j0b + o);
            sum += wo[1] * s1 + wo[2] * ((1.0 / 3.0) * s2);
          }
          sum *= W[3 * (direct ? (size_t)q * NB + j0b + m : (size_t)k1 * NB + m)] * s_down[t % nT];
          if (!a.mirror) {
            if (nS == 1) {
              dir += sum;
            } else {
              double& out = a.partial[((size_t)item * J + m) * nS + t];
              out = (k1 == k1_first ? 0.0 : out) + sum;
            }
          } else {
            a.partial[((direct ? slot : mslot) * NB + m) * nS + t] = sum;
          }
          if constexpr (SL) {
            if (!unit) {
              // bound of the weak terms at their block's scale; the order of these additions decides no bit of a rate
              double weak = 0.0;
              for (int o = 0; o < (direct ? NB : J); ++o) {
                const int ab = (direct ? m : o) * NB + (direct ? o : m);
                auto bound = [&](int k) {
                  const int* wk = sWeak + (k * J * NB + ab) * (nS + 1);
                  return wk[t] ? wk[nS] * __hiloint2double(wk[t] + 1, 0) : 0.0;
                };
                const double w1 = bound(0), w2 = bound(direct ? 1 : 2);
                const double* wo = W + 3 * (direct ? (size_t)k1 * NB + o : (size_t)q * NB + j0b + o);
                if (w1 > 0.0 || w2 > 0.0) weak += (wo[1] * w1 + wo[2] * ((1.0 / 3.0) * w2)) * scalbn(1.0, 2 * sSc[ab]);
              }
              if (weak > 0.0)
                atomicAdd(a.weak + (size_t)t * NM + (direct ? (size_t)q * NB + j0b + m : (size_t)rq * NB + m),
                          weak * W[3 * (direct ? (size_t)q * NB + j0b + m : (size_t)k1 * NB + m)] * s_down[t % nT]);
            }
          }
        }
        __syncthreads();
      }
      if (a.item_counts) {
        unsigned* sCnt = reinterpret_cast<unsigned*>(sRed);
        if (has_row) {
          sCnt[tid] = n1 + n4;
          sCnt[rows + tid] = n1 + n5;
        }
        __syncthreads();
        if (tid < nout) {
          const bool direct = tid < J;
          const int m = direct ? tid : tid - J;
          unsigned long long sum = 0;
          for (int r = 0; r < (direct ? NB2 : J * NB); ++r)
            sum += direct ? sCnt[m * NB2 + r] : sCnt[rows + (r / NB) * NB2 + m * NB + r % NB];
          if (!a.mirror)
            dir_n += sum;
          else
            a.item_counts[(direct ? slot : mslot) * NB + m] = sum;
        }
        __syncthreads();
      }
    }
    if (!a.mirror && tid < J) {
      if (nS == 1)
        a.partial[(size_t)item * J + tid] = dir;
      else if (k1_first >= k1_end)
        for (int t = 0; t < nS; ++t) a.partial[((size_t)item * J + tid) * nS + t] = 0.0;
      if (a.item_counts) a.item_counts[(size_t)item * J + tid] = dir_n;
    }
    unsigned long long c0 = cnt0, c1 = cnt1, c2 = cnt2, cw = nwf, ct = nte;
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
      if (tid == 0 && niter) {
        atomicAdd(a.counts + 6, niter);
        atomicAdd(a.counts + 7, npair);
      }
    }
  }
}

}  // namespace
}  // namespace fp

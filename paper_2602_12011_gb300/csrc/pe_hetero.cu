// pe_hetero.cu -- heterodyned (relative-binning) log-likelihood (the heterodyning idea of Sec. 1,
// in the per-mode relative-binning form of Zackay, Dai & Venumadhav 2018 / Leslie, Dai & Pratten
// 2021): host edge construction, summary-data kernels and the per-sample kernel, plus the C ABI.
//
//   k_mode_brackets  reference per-mode A/E/T brackets on the fine bins [0, K) (creation)
//   k_het_summary    per coarse bin: A_o (o = 0, 1) and B_o (o = 0, 1, 2) by sequential sums
//   k_het_loglike    one CTA per sample: ratios at every edge of every detector (shared memory),
//                    then the per-bin contraction and a fixed-order block reduction
//
// The brackets B_c (A/E/T combinations of X', Y', Z' before the factor Q n_c) stand for the channel
// signals: ratios are the same, and dg = conj(d) w Q n_c, gg = w |Q|^2 n_c^2 supply the rest.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <set>
#include <vector>

#include "pe_device.cuh"
#include "pe_device_fx.cuh"
#include "pe_device_mixed.cuh"
#include "pe_internal.h"
#include "pe_kernels.h"
#include "pespace_gb300.h"
#include "pe_fault.h"

namespace pe {

constexpr int kHetMaxEdges = 640;
constexpr int kHetThreads = 320;   // most threads of a CTA of k_het_loglike
// Threads of a detector with ne edges: equal rounds of edges over the fewest threads (at least 64, which stage the projection forms). They
// also share out its bins, so the order of its sums depends on nothing but its own edges; a CTA has those of the detector that wants the most.
inline int het_threads(int ne) {
  const int rounds = (ne + kHetThreads - 1) / kHetThreads, t = ((ne + rounds - 1) / rounds + 31) / 32 * 32;
  return t < 64 ? 64 : t;
}
constexpr int kPairs = kNModes * (kNModes + 1) / 2;   // unordered mode pairs (md <= md2)

__host__ __device__ constexpr int pair_index(int a, int b) {   // a <= b
  return a * kNModes - a * (a - 1) / 2 + (b - a);
}

struct HetDev {
  DetDev det;
  const int* edge;       // [ne] fine-bin indices
  const double* fe;      // [ne] edge frequencies
  const double2* ih0e;   // [ne][5][3] inverses 1/h0 of the reference brackets at the edges (0 where h0 = 0)
  const int* src;        // [ne][5][3] edge whose ratio applies (carry-forward), -1 for none
  const double2* A;      // [5][3][2][ne-1]: consecutive bins are consecutive, for the contraction's loads
  const double2* Bs;     // [kPairs][3][3][ne-1]
  const float4* Aw;      // A and Bs over the edges' ratios, in double words, for the mixed kernel (k_het_dw)
  const float4* Bw;
  const longlong2* Ax;   // A and Bs for the fixed-point contraction (k_het_words): packed words of re, im
  const longlong2* Bx;
  const int* Gx;         // [6][3][ne-1] their exponents
  int ne;
  int nt;                // threads that share out its bins (het_threads)
  unsigned mask;
};
struct HetSet {
  HetDev h[kMaxDet];
  int n;
  int nemax;   // largest ne of the set (rows of the kernel's ratio table)
};

__device__ __forceinline__ double2 cconj(double2 a) { return make_double2(a.x, -a.y); }

// Per-mode brackets of one sample at bin b (zero for inactive modes or bins past a mode's end).
__device__ __forceinline__ void mode_brackets(const DetDev& D, const SampleCoef& S, int b, unsigned mask,
                                              double2 o[kNModes][3], const double2* __restrict__ tab,
                                              const double* __restrict__ pc) {
  BinIn Bn;
  load_bin(D, b, S.tc, Bn);
#pragma unroll 1
  for (int md = 0; md < kNModes; ++md) {
    const ModeCoef& C = S.md[md];
    XYZAcc a;
    xyz_zero(a);
    if ((mask >> md) & 1u && C.active && Bn.f < C.fend) mode_bin(D, S, C, Bn, a, tab, pc);
    double2 x[3];
    xyz_final(a, Bn.z, x);
    aet_from_xyz(x, o[md]);
  }
}

// The same with the fixed-point unit (STRIDE: threads of the CTA, between the entries of a column).
template <int STRIDE>
__device__ __forceinline__ void mode_brackets_fx(const DetDev& D, const SampleCoef& S, int b, unsigned mask,
                                                 double2 o[kNModes][3], const DetDev& D0,
                                                 const fx* __restrict__ pc, fx* col) {
  FxBin Bn;
  load_bin_fx(D, b, S.tc, Bn);
  const double2 z = D.z[b];
#pragma unroll 1
  for (int md = 0; md < kNModes; ++md) {
    const ModeCoef& C = S.md[md];
    FxAccT<STRIDE> a;
    fx_zero(a, col);
    if ((mask >> md) & 1u && C.active && Bn.f < C.fend) mode_bin_fx(D, S, C, Bn, a, D0.fcis, D0.fsinc, pc, md);
    aet_from_fx(a, z, o[md]);
  }
}

// The same with the mixed-precision unit (FP64 phase, t_f and turn reductions; double-word
// geometry), each mode's brackets returned to FP64.
__device__ __forceinline__ void mode_brackets_mixed(const DetDev& D, const SampleCoef& S, int b, unsigned mask,
                                                    double2 o[kNModes][3], const float4* __restrict__ tab,
                                                    const float2* __restrict__ pcw) {
  BinIn Bn;
  load_bin(D, b, S.tc, Bn);
  BinW W;
  load_bin_w(D, b, W);
  const float4 zz = D.zw[b];
  const cdf z = {df_make(zz.x, zz.y), df_make(zz.z, zz.w)};
#pragma unroll 1
  for (int md = 0; md < kNModes; ++md) {
    const ModeCoef& C = S.md[md];
    MixAcc a;
    mix_zero(a);
    if ((mask >> md) & 1u && C.active && Bn.f < C.fend) mode_bin_mixed(D, S, C, Bn, W, a, tab, pcw);
    cdf x[3], od[3];
    mix_final(a, z, x);
    aet_from_xyz_dw(x, od);
    for (int c = 0; c < 3; ++c) o[md][c] = make_double2(df_to(od[c].re) * S.ihsc, df_to(od[c].im) * S.ihsc);
  }
}

// Reference per-mode brackets on bins [0, K): out[(md*3 + c)*K + k].
template <bool FX>
__global__ void k_mode_brackets(DetDev D, const SampleCoef* coef, int K, unsigned mask, double2* out) {
  __shared__ __align__(16) double pc[kFxProj];
  __shared__ fx fxcol[FX ? kFxSums : 1][kTileBins];
  const SampleCoef& S = coef[0];
  if (FX)
    fx_proj_prologue(D, S, reinterpret_cast<fx*>(pc));
  else
    proj_prologue(D, S, pc);
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= K) return;
  double2 o[kNModes][3];
  if (FX)
    mode_brackets_fx<kTileBins>(D, S, k, mask, o, D, reinterpret_cast<const fx*>(pc), &fxcol[0][threadIdx.x]);
  else
    mode_brackets(D, S, k, mask, o, D.sct, pc);
  for (int md = 0; md < kNModes; ++md)
    for (int c = 0; c < 3; ++c) out[((size_t)md * 3 + c) * K + k] = o[md][c];
}

// h0e[(i*5 + md)*3 + c] = reference bracket (md, c) at edge i
__global__ void k_gather_edges(const double2* hb, int K, const int* edge, int ne, double2* h0e) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= ne * kNModes * 3) return;
  const int i = j / (kNModes * 3), mc = j % (kNModes * 3);
  h0e[j] = hb[(size_t)mc * K + edge[i]];
}

// h0e -> 1/h0e in place; 0 where |h0e|^2 is 0 (h0e = 0, never a ratio source, or so small that its
// square underflows, where the ratio becomes 0 instead of the overflow a division would give)
__global__ void k_invert_edges(double2* h0e, int n) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const double2 h = h0e[j];
  const double den = h.x * h.x + h.y * h.y;
  h0e[j] = den != 0.0 ? make_double2(h.x / den, -h.y / den) : make_double2(0.0, 0.0);
}

// Summary data: one thread per (coarse bin, quantity); a sequential sum over the bin's fine bins.
// Quantities per bin: A: 5 modes x 3 channels x 2 orders; B: kPairs x 3 x 3 orders.
__global__ void k_het_summary(DetDev D, const int* edge, const double* fe, int ne, const double2* h0, int K,
                              double2* A, double2* Bs) {
  constexpr int nA = kNModes * 3 * 2, nB = kPairs * 3 * 3;
  const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int nbin = ne - 1;
  if (id >= (long long)nbin * (nA + nB)) return;
  const int b = (int)(id / (nA + nB)), q = (int)(id % (nA + nB));
  const int lo = edge[b], hi = edge[b + 1] + (b == nbin - 1 ? 1 : 0);
  double2 acc = make_double2(0.0, 0.0);
  if (q < nA) {
    const int md = q / 6, c = (q / 2) % 3, o = q % 2;
    const double2* h = h0 + ((size_t)md * 3 + c) * K;
    for (int k = lo; k < hi; ++k) {
      const double df = D.f[k] - fe[b];
      const double2 t = cmul(D.dg[c * D.nb + k], h[k]);   // conj(d) w Q n_c B0
      const double s = (o == 0) ? 1.0 : df;
      acc.x = fma(t.x, s, acc.x);
      acc.y = fma(t.y, s, acc.y);
    }
    A[(size_t)((md * 3 + c) * 2 + o) * nbin + b] = acc;
  } else {
    const int r = q - nA;
    const int p = r / 9, c = (r / 3) % 3, o = r % 3;
    int m1 = 0, m2 = 0;
    for (int a = 0; a < kNModes; ++a)
      for (int bb = a; bb < kNModes; ++bb)
        if (pair_index(a, bb) == p) { m1 = a; m2 = bb; }
    const double2* h1 = h0 + ((size_t)m1 * 3 + c) * K;
    const double2* h2 = h0 + ((size_t)m2 * 3 + c) * K;
    for (int k = lo; k < hi; ++k) {
      const double df = D.f[k] - fe[b];
      const double s = D.gg[c * D.nb + k] * (o == 0 ? 1.0 : (o == 1 ? df : df * df));
      const double2 t = cmul(h1[k], cconj(h2[k]));
      acc.x = fma(t.x, s, acc.x);
      acc.y = fma(t.y, s, acc.y);
    }
    Bs[(size_t)((p * 3 + c) * 3 + o) * nbin + b] = acc;
  }
}

// Summary data of one (channel c, bin b) for the mixed contraction, over the ratios at the bin's two edges: with slopes
// (rb - ra) / (fe[b+1] - fe[b]) the moments A0, A1 become A_a = A0 - A1', A_b = A1' and B0, B1, B2 become
// B_aa = B0 - 2 B1' + B2', B_ab = B1' - B2', B_bb = B2' (primes: over the width's powers), as double words (re hi, re lo, im hi, im lo).
__global__ void k_het_dw(const double* fe, int ne, const double2* A, const double2* Bs, float4* Aw, float4* Bw) {
  const int nbin = ne - 1, i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 3 * nbin) return;
  const int c = i / nbin, b = i % nbin;
  const double idf = 1.0 / (fe[b + 1] - fe[b]);
  auto put = [](float4* o, double x, double y) {
    const float2 re = to_dw(x), im = to_dw(y);
    *o = make_float4(re.x, re.y, im.x, im.y);
  };
  for (int md = 0; md < kNModes; ++md) {
    const size_t r = (size_t)(md * 3 + c) * 2 * nbin + b;
    const double2 a0 = A[r], a1 = make_double2(A[r + nbin].x * idf, A[r + nbin].y * idf);
    put(Aw + r, a0.x - a1.x, a0.y - a1.y);
    put(Aw + r + nbin, a1.x, a1.y);
  }
  for (int pr = 0; pr < kPairs; ++pr) {
    const size_t r = (size_t)(pr * 3 + c) * 3 * nbin + b;
    const double2 b0 = Bs[r], b1 = make_double2(Bs[r + nbin].x * idf, Bs[r + nbin].y * idf);
    const double2 b2 = make_double2(Bs[r + 2 * nbin].x * idf * idf, Bs[r + 2 * nbin].y * idf * idf);
    put(Bw + r, (b0.x - b1.x) - (b1.x - b2.x), (b0.y - b1.y) - (b1.y - b2.y));
    put(Bw + r + nbin, b1.x - b2.x, b1.y - b2.y);
    put(Bw + r + 2 * nbin, b2.x, b2.y);
  }
}

__device__ __forceinline__ cdf unpack4(float4 q) { return cdf{df_make(q.x, q.y), df_make(q.z, q.w)}; }

// Ratios the mixed kernel keeps as double words stay below this magnitude. Normal ratios are O(1);
// one far larger comes only from an edge where the reference signal has almost vanished (a tapered
// end that the sample outlives), and a bin that uses such an edge is contracted in FP64 instead
// (ratio squares times 1/df^2 stay far inside the FP32 exponent range below it).
constexpr double kHetDwRatioMax = 16777216.0;   // 2^24

// FP64 contraction of coarse bin b, channel c: (<d|h>, <h|h>) from the ratios ld(edge, md) and the
// summary data A, B.
template <class Ld>
__device__ __forceinline__ void het_bin_fp64(const HetDev& H, int b, int c, Ld ld, double& dh, double& hh) {
  const double idf = 1.0 / (H.fe[b + 1] - H.fe[b]);
  double2 r0[kNModes], r1[kNModes];
  for (int md = 0; md < kNModes; ++md) {
    const int s0 = H.src[(b * kNModes + md) * 3 + c], s1 = H.src[((b + 1) * kNModes + md) * 3 + c];
    const double2 ra = s0 >= 0 ? ld(s0, md) : make_double2(0.0, 0.0);
    const double2 rb = s1 >= 0 ? ld(s1, md) : make_double2(0.0, 0.0);
    r0[md] = ra;
    r1[md] = make_double2((rb.x - ra.x) * idf, (rb.y - ra.y) * idf);
  }
  // <h|h> = Re sum_i [ r0_i sum_j (B0_ij r0_j* + B1_ij r1_j*) + r1_i sum_j (B1_ij r0_j* + B2_ij r1_j*) ], off-diagonal pairs
  // (j > i) twice: 16 FMAs a pair and 4 a mode, against 26 a pair for the products t0, t1, t2 of the ratios
  const int nbin = H.ne - 1;
  dh = 0.0;
  hh = 0.0;
#pragma unroll
  for (int md = 0; md < kNModes; ++md) {
    const double2* a = H.A + (size_t)(md * 3 + c) * 2 * nbin + b;
    const double2 a0 = a[0], a1 = a[nbin];
    dh = fma(a0.x, r0[md].x, fma(-a0.y, r0[md].y, fma(a1.x, r1[md].x, fma(-a1.y, r1[md].y, dh))));
    double2 y = make_double2(0.0, 0.0), w = y;
#pragma unroll
    for (int k = 1; k <= kNModes; ++k) {
      const int m2 = k < kNModes ? (md + k) : md;   // the off-diagonal pairs first, doubled, then the diagonal one
      if (m2 >= kNModes) continue;
      if (k == kNModes) { y.x *= 2.0; y.y *= 2.0; w.x *= 2.0; w.y *= 2.0; }
      const double2* q = H.Bs + (size_t)(pair_index(md, m2) * 3 + c) * 3 * nbin + b;
      const double2 q0 = q[0], q1 = q[nbin], q2 = q[2 * nbin];
      const double2 s0 = r0[m2], s1 = r1[m2];
      y.x = fma(q0.x, s0.x, fma(q0.y, s0.y, fma(q1.x, s1.x, fma(q1.y, s1.y, y.x))));
      y.y = fma(q0.y, s0.x, fma(-q0.x, s0.y, fma(q1.y, s1.x, fma(-q1.x, s1.y, y.y))));
      w.x = fma(q1.x, s0.x, fma(q1.y, s0.y, fma(q2.x, s1.x, fma(q2.y, s1.y, w.x))));
      w.y = fma(q1.y, s0.x, fma(-q1.x, s0.y, fma(q2.y, s1.x, fma(-q2.x, s1.y, w.y))));
    }
    hh = fma(r0[md].x, y.x, fma(-r0[md].y, y.y, fma(r1[md].x, w.x, fma(-r1[md].y, w.y, hh))));
  }
}
// Summary data of one (channel c, bin b) for the fixed-point contraction (het_bin_fx), over ra and d = rb - ra (the slopes'
// powers of 1/(fe[b+1] - fe[b]) in the data). Every mode is scaled by 2^-g, the least power of two above its
// sqrt(B0_ii), the norm of its reference signal in the bin; with that the entries of Bs are below 1 (Cauchy-Schwarz) and are
// words in 2^-60, and those of A are below 2^a, words in 2^(a - 60); packed for multiplication (fx_pack). Gx: rows 0..4
// the g, row 5 a. A bin whose data the words cannot hold (an inf or NaN, a norm outside 2^+-400, entries of a
// mode without a norm) has a = kHetGeneral and is contracted in FP64.
constexpr int kHetGeneral = 1 << 20;
constexpr int kHetNoMode = -(1 << 20);   // g of a mode without signal in the bin
constexpr int kHetExpo = 450;            // bound of the exponents a and N (het_bin_fx)
constexpr int kHetLeast = 50;            // least hh of the fixed-point form, 2^kHetLeast in 2^-60
__global__ void k_het_words(const double* fe, int ne, const double2* A, const double2* Bs, longlong2* Ax, longlong2* Bx, int* Gx) {
  const int nbin = ne - 1, i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 3 * nbin) return;
  const int c = i / nbin, b = i % nbin;
  const double idf = 1.0 / (fe[b + 1] - fe[b]);
  auto at = [&](const double2* q, int row, int o) {
    const double2 v = q[(size_t)row * nbin + b];
    const double f = o == 0 ? 1.0 : (o == 1 ? idf : idf * idf);
    return make_double2(v.x * f, v.y * f);
  };
  auto row_a = [&](int md, int o) { return (md * 3 + c) * 2 + o; };
  auto row_b = [&](int pr, int o) { return (pr * 3 + c) * 3 + o; };
  auto mag = [](double2 v) { return fabs(v.x) > fabs(v.y) || isnan(v.x) ? fabs(v.x) : fabs(v.y); };   // NaN if either is one
  int g[kNModes], a = -kHetGeneral;
  bool ok = true;
  for (int md = 0; md < kNModes; ++md) {
    const double n2 = at(Bs, row_b(pair_index(md, md), 0), 0).x;
    const bool some = n2 > 0x1p-800 && n2 < 0x1p800;
    g[md] = some ? (fx_expo(n2) - 1021) >> 1 : kHetNoMode;     // n2 < 2^(2 g), and >= 2^(2 g - 2)
    for (int o = 0; o < 2; ++o) {
      const double m = mag(at(A, row_a(md, o), o));
      if (some && m > 0.0) a = max(a, fx_expo(m) - 1022 - g[md]);
      ok &= some ? m < 0x1p800 : m == 0.0;
    }
  }
  if (a == -kHetGeneral) a = 0;
  ok &= a > -kHetExpo && a < kHetExpo;
  auto word = [](double2 v, int e) {   // v 2^-e, rounded
    auto q = [&](double x) { return fx_pack(fx_split((fx_from_bits(scalbn(x, -e), 61) + 1) >> 1)); };
    return longlong2{q(v.x), q(v.y)};
  };
  for (int m1 = 0; m1 < kNModes; ++m1)
    for (int m2 = m1; m2 < kNModes; ++m2)
      for (int o = 0; o < 3; ++o) {
        const int r = row_b(pair_index(m1, m2), o);
        const double2 v = at(Bs, r, o);
        const bool some = g[m1] != kHetNoMode && g[m2] != kHetNoMode;
        const int e = some ? g[m1] + g[m2] : 0;
        const bool in = some ? mag(v) <= scalbn(1.0625, e) : mag(v) == 0.0;
        ok &= in;
        Bx[(size_t)r * nbin + b] = in ? word(v, e) : longlong2{0, 0};
      }
  for (int md = 0; md < kNModes; ++md) {
    for (int o = 0; o < 2; ++o)
      Ax[(size_t)row_a(md, o) * nbin + b] = ok && g[md] != kHetNoMode ? word(at(A, row_a(md, o), o), g[md] + a) : longlong2{0, 0};
    Gx[(size_t)(md * 3 + c) * nbin + b] = g[md];
  }
  Gx[(size_t)(kNModes * 3 + c) * nbin + b] = ok ? a : kHetGeneral;
}

// het_bin_fp64's contraction in fixed point, block floating per (bin, channel): with m_i the largest component of mode i's
// ratios at the two edges, every ratio is held in 2^-60 of 2^(N - g_i), N the least power of two for which sum m_i 2^(g_i - N)
// is below 1/2. What is lost is then below 2^-59 of the sample's own signal in the bin, whatever its distance
// and however the modes' ratios differ (FP64 keeps 2^-53 of each ratio), and powers of two in the signal pass through exactly.
// Bounds: d is below 1, y and w below sqrt(2) (Cauchy-Schwarz over the bin's fine bins), hh below 1/2 and, where neither the modes nor
// the edges cancel, above 2^-8. False where the bin takes the FP64 form: a ratio that is not finite, exponents outside the words', or an edge whose
// ratio is far above the signal in the bin (the reference has almost vanished there): a mode's ratios differ fourfold or more and hh is
// below 2^-10. Where hh is that small because the terms cancel, FP64 loses more. (A bin left to the FP64 form costs its CTA some 30 us: its 340
// operations are one thread's chain. With every hh below 2^-10 left to it, a bin or two in a sample, calls took 5 to 9 % longer.)
// Bound by the 32 x 32-bit products, about 900 per (bin, channel) at 16 per SM and clock where the FP64 form issues 340 operations
// at 1.67 (777 samples, LISA, 2^22 s, whole call: 677 us with the FP64 form, 356 us at any distance; 363 us, and 749 at a third of the reference's distance, with the ratios
// held in 2^-59 of 1, which lost the faint samples' bits and sent ratios above 2 to the FP64 form).
__device__ __forceinline__ bool het_bin_fx(const HetDev& H, int b, int c, const double2* __restrict__ ratio, double& dh, double& hh) {
  const int nbin = H.ne - 1;
  const int ea = H.Gx[(size_t)(kNModes * 3 + c) * nbin + b];
  if (ea == kHetGeneral) return false;
  const int *sa = H.src + (size_t)b * kNModes * 3 + c, *sb = sa + kNModes * 3;
  auto at = [&](int e, int md) { return e >= 0 ? ratio[(e * kNModes + md) * 3 + c] : make_double2(0.0, 0.0); };
  unsigned m[kNModes];
  int g[kNModes], top = 2 * kHetNoMode;
  unsigned most = 0;
  bool uneven = false;                    // a mode's ratios differ fourfold or more
#pragma unroll
  for (int md = 0; md < kNModes; ++md) {
    const double2 ra = at(sa[3 * md], md), rb = at(sb[3 * md], md);
    auto hi = [](double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; };
    const unsigned ma = max(hi(ra.x), hi(ra.y)), mb = max(hi(rb.x), hi(rb.y));
    m[md] = max(ma, mb);
    uneven |= m[md] - min(ma, mb) >= 0x200000u;
    g[md] = H.Gx[(size_t)(md * 3 + c) * nbin + b];
    most = max(most, m[md]);
    if (m[md] >= 0x100000u) top = max(top, (int)(m[md] >> 20) + g[md]);
  }
  dh = 0.0;
  hh = 0.0;
  if (most < 0x100000u) return true;      // no ratio (or none above 2^-1022)
  if (most >= 0x7ff00000u) return false;
  unsigned sum = 0;                       // above sum m_i 2^g_i, in 2^(top - 1043)
#pragma unroll
  for (int md = 0; md < kNModes; ++md)
    if (m[md] >= 0x100000u) sum += (((m[md] & 0xfffffu) | 0x100000u) >> min(top - (int)(m[md] >> 20) - g[md], 31)) + 1;
  const int N = top - 1043 + (32 - __clz(sum)) + 1;
  if (N < -kHetExpo || N > kHetExpo) return false;
  fxs rr[kNModes], ri[kNModes], dr[kNModes], di[kNModes];
#pragma unroll
  for (int md = 0; md < kNModes; ++md) {
    const double2 ra = at(sa[3 * md], md), rb = at(sb[3 * md], md);
    const int k = 60 + g[md] - N;
    const fx ax = fx_from_bits(ra.x, k), ay = fx_from_bits(ra.y, k);
    rr[md] = fx_split(ax);
    ri[md] = fx_split(ay);
    dr[md] = fx_split(fx_from_bits(rb.x, k) - ax);
    di[md] = fx_split(fx_from_bits(rb.y, k) - ay);
  }
  fx sd = 0, sh = 0;
#pragma unroll
  for (int md = 0; md < kNModes; ++md) {
    const longlong2* a = H.Ax + (size_t)(md * 3 + c) * 2 * nbin + b;
    const longlong2 w0 = a[0], w1 = a[nbin];
    sd += fx_msub(fx_unpack(w0.x), rr[md], fx_unpack(w0.y), ri[md]) + fx_msub(fx_unpack(w1.x), dr[md], fx_unpack(w1.y), di[md]);
    fx yx = 0, yy = 0, wx = 0, wy = 0;
#pragma unroll
    for (int k = 1; k <= kNModes; ++k) {
      const int m2 = k < kNModes ? (md + k) : md;   // the off-diagonal pairs first, doubled, then the diagonal one
      if (m2 >= kNModes) continue;
      if (k == kNModes) { yx *= 2; yy *= 2; wx *= 2; wy *= 2; }
      const longlong2* q = H.Bx + (size_t)(pair_index(md, m2) * 3 + c) * 3 * nbin + b;
      const longlong2 u0 = q[0], u1 = q[nbin], u2 = q[2 * nbin];
      const fxs x0 = fx_unpack(u0.x), y0 = fx_unpack(u0.y), x1 = fx_unpack(u1.x), y1 = fx_unpack(u1.y), x2 = fx_unpack(u2.x), y2 = fx_unpack(u2.y);
      // (x + i y) conj(r): (x rr + y ri) + i (y rr - x ri)
      auto madd = [&](fxs a0, fxs b0, fxs a1, fxs b1, fxs a2, fxs b2, fxs a3, fxs b3) {
        fxa t = fx_prod<4>(a0, b0);
        fx_mac(t, a1, b1);
        fx_mac(t, a2, b2);
        fx_mac(t, a3, b3);
        return fx_val(t);
      };
      auto msub = [&](fxs a0, fxs b0, fxs a1, fxs b1, fxs a2, fxs b2, fxs a3, fxs b3) {   // a0 b0 + a1 b1 - a2 b2 - a3 b3
        fxa t = fx_prod<0>(a0, b0), n = fxa{fx_mulw(a2.h, b2.h), fx_madw(a2.h, b2.l, fx_mulw(a2.l, b2.h))};
        fx_mac(t, a1, b1);
        fx_mac(n, a3, b3);
        return (t.h - n.h) + ((t.c - n.c) >> 30);
      };
      yx += madd(x0, rr[m2], y0, ri[m2], x1, dr[m2], y1, di[m2]);
      yy += msub(y0, rr[m2], y1, dr[m2], x0, ri[m2], x1, di[m2]);
      wx += madd(x1, rr[m2], y1, ri[m2], x2, dr[m2], y2, di[m2]);
      wy += msub(y1, rr[m2], y2, dr[m2], x1, ri[m2], x2, di[m2]);
    }
    sh += fx_msub(rr[md], fx_split(yx), ri[md], fx_split(yy)) + fx_msub(dr[md], fx_split(wx), di[md], fx_split(wy));
  }
  if (uneven && sh < (1LL << kHetLeast)) return false;
  dh = fx_to_double(sd, ea + N - 60);
  hh = fx_to_double(sh, 2 * N - 60);
  return true;
}

// Re(a b) and Re(a conj(b)) in double words
__device__ __forceinline__ df re_mul(const cdf& a, const cdf& b) { return dfl_sub(dfl_mul(a.re, b.re), dfl_mul(a.im, b.im)); }
__device__ __forceinline__ cdf mul_conj(const cdf& a, const cdf& b) {
  return cdf{dfl_add(dfl_mul(a.re, b.re), dfl_mul(a.im, b.im)), dfl_sub(dfl_mul(a.im, b.re), dfl_mul(a.re, b.im))};
}

// Block sum of six doubles per thread in a fixed tree order (up to kHetThreads threads); result valid in thread 0.
__device__ __forceinline__ void het_block_sum(double v[6], double (*sh)[kHetThreads / 32]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_down_sync(0xffffffffu, v[i], o);
    if (lane == 0) sh[i][wid] = v[i];
  }
  __syncthreads();
  if (threadIdx.x == 0)
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      v[i] = 0.0;
      for (int w = 0; w < nw; ++w) v[i] += sh[i][w];
    }
}

// One CTA per sample. Dynamic shared memory: [max ne][5][3] double2 ratios, which fits two CTAs on an SM at the default 300
// edges; so a CTA has a thread for (nearly) every edge, up to kHetThreads: with 128 threads an SM had eight warps
// and three rounds of edges, the last a third full (777 samples, LISA: 1.09 ms).
// The signal at the edges comes from the fixed-point unit (FX; both precisions), or the precision's own where a detector
// does not take that unit. MIX: the ratios are kept as double words and contracted in double words (Aw, Bw);
// the sums across bins and the block reduction stay FP64. An edge with a ratio of kHetDwRatioMax or more
// keeps all its ratios in FP64 (flag byte per edge after the ratios), and every (bin, channel) that reads it
// takes the FP64 contraction. FP64 on the fixed-point unit: the ratios stay FP64, and the contraction holds them in
// fixed point relative to the bin's largest (het_bin_fx).
template <bool MIX, bool FX>
__global__ void __launch_bounds__(kHetThreads, 2) k_het_loglike(HetSet hs, int B, const SampleCoef* __restrict__ coef,
                                                               double* logl, double* dhhh) {
  extern __shared__ double2 rsh[];
  unsigned char* wflag = reinterpret_cast<unsigned char*>(rsh + (size_t)hs.nemax * kNModes * 3);
  constexpr bool DW = MIX && !FX;   // the mixed unit at the edges
  constexpr bool XC = FX && !MIX;   // the fixed-point contraction
  __shared__ __align__(16) double pc[kFxProj];
  __shared__ float2 pcw[DW ? kProj : 1];
  __shared__ double sh[6][kHetThreads / 32];
  __shared__ double2 stab[DW || FX ? 1 : kSinTab];
  __shared__ fx fxcol[FX ? kFxSums : 1][kHetThreads];
  __shared__ float4 stabw[DW ? kSinTab : 1];
  if constexpr (DW) {
    for (int i = threadIdx.x; i < kSinTab; i += blockDim.x) stabw[i] = hs.h[0].det.sctw[i];
  } else if constexpr (!FX) {
    for (int i = threadIdx.x; i < kSinTab; i += blockDim.x) stab[i] = hs.h[0].det.sct[i];
  }
  const int s = blockIdx.x;
  const SampleCoef& S = coef[s];
  double L = 0.0;
  for (int I = 0; I < hs.n; ++I) {
    const HetDev& H = hs.h[I];
    const DetDev& D = H.det;
    // its barriers also order the table staging and the previous detector
    if constexpr (FX)
      fx_proj_prologue(D, S, reinterpret_cast<fx*>(pc));
    else
      proj_prologue(D, S, pc);
    if constexpr (DW) {
      if (threadIdx.x < kProj) pcw[threadIdx.x] = to_dw(pc[threadIdx.x]);
      __syncthreads();
    }
    for (int e = threadIdx.x; e < H.ne; e += blockDim.x) {
      bool need = false;
      for (int j = 0; j < kNModes * 3; ++j) need |= (H.src[e * kNModes * 3 + j] == e);
      if (!need) continue;
      double2 o[kNModes][3];
      if constexpr (DW)
        mode_brackets_mixed(D, S, H.edge[e], H.mask, o, stabw, pcw);
      else if constexpr (FX)
        mode_brackets_fx<kHetThreads>(D, S, H.edge[e], H.mask, o, hs.h[0].det, reinterpret_cast<const fx*>(pc), &fxcol[0][threadIdx.x]);
      else
        mode_brackets(D, S, H.edge[e], H.mask, o, stab, pc);
      // ratios in place of the brackets; in the mixed kernel, flag the edge if one of them is out
      // of the double words' range (also for inf and NaN)
      bool wide = false;
#pragma unroll
      for (int md = 0; md < kNModes; ++md)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const int j = (e * kNModes + md) * 3 + c;
          if (H.src[j] != e) continue;
          o[md][c] = cmul(o[md][c], H.ih0e[j]);
          if constexpr (MIX) wide |= !(fmax(fabs(o[md][c].x), fabs(o[md][c].y)) < kHetDwRatioMax);
        }
      if constexpr (MIX) wflag[e] = wide ? 1 : 0;
#pragma unroll
      for (int md = 0; md < kNModes; ++md)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const int j = (e * kNModes + md) * 3 + c;
          if (H.src[j] != e) continue;
          if (MIX && !wide) {
            const float2 re = to_dw(o[md][c].x), im = to_dw(o[md][c].y);
            reinterpret_cast<float4*>(rsh)[j] = make_float4(re.x, re.y, im.x, im.y);
          } else {
            rsh[j] = o[md][c];
          }
        }
    }
    __syncthreads();
    double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    if constexpr (MIX) {
      // double words over the ratios at both edges, in rolled loops that read the ratios from shared memory: unrolled over the pairs
      // the code overran the instruction cache (3.79 -> 3.76 ms, 4096 samples on two detectors)
      const float4* rw = reinterpret_cast<const float4*>(rsh);
      const cdf zc = {df_make(0.f, 0.f), df_make(0.f, 0.f)};
      const int nbin = H.ne - 1;
      for (int b = threadIdx.x < H.nt ? threadIdx.x : nbin; b < nbin; b += H.nt) {
#pragma unroll 1
        for (int c = 0; c < 3; ++c) {
          const int* sa = H.src + (size_t)b * kNModes * 3 + c;          // edge of mode md's ratio at sa[3 md], and at the
          const int* sb = sa + kNModes * 3;                             // bin's other edge
          bool wide = false;
#pragma unroll
          for (int md = 0; md < kNModes; ++md) {
            const int s0 = sa[3 * md], s1 = sb[3 * md];
            wide |= (s0 >= 0 && wflag[s0]) || (s1 >= 0 && wflag[s1]);
          }
          if (wide) {   // an edge of this bin keeps FP64 ratios
            auto ld = [&](int e, int md) -> double2 {
              const int j = (e * kNModes + md) * 3 + c;
              if (wflag[e]) return rsh[j];
              const cdf r = unpack4(rw[j]);
              return make_double2(df_to(r.re), df_to(r.im));
            };
            double dh, hh;
            het_bin_fp64(H, b, c, ld, dh, hh);
            v[c] += dh;
            v[3 + c] += hh;
            continue;
          }
          auto ratio = [&](int e, int md) { return e >= 0 ? unpack4(rw[(e * kNModes + md) * 3 + c]) : zc; };
          df dh = df_make(0.f, 0.f), hh = df_make(0.f, 0.f);
#pragma unroll 1
          for (int md = 0; md < kNModes; ++md) {
            const cdf ra = ratio(sa[3 * md], md), rb = ratio(sb[3 * md], md);
            const float4* a = H.Aw + (size_t)(md * 3 + c) * 2 * nbin + b;
            dh = dfl_add(dh, dfl_add(re_mul(unpack4(a[0]), ra), re_mul(unpack4(a[nbin]), rb)));
            cdf y = zc, w = zc;
#pragma unroll 1
            for (int m2 = kNModes - 1; m2 >= md; --m2) {   // the off-diagonal pairs first, doubled, then the diagonal one
              if (m2 == md) {
                y = cdf{df_scale2(y.re, 2.f), df_scale2(y.im, 2.f)};
                w = cdf{df_scale2(w.re, 2.f), df_scale2(w.im, 2.f)};
              }
              const cdf la = ratio(sa[3 * m2], m2), lb = ratio(sb[3 * m2], m2);
              const float4* q = H.Bw + (size_t)(pair_index(md, m2) * 3 + c) * 3 * nbin + b;
              const cdf q0 = unpack4(q[0]), q1 = unpack4(q[nbin]), q2 = unpack4(q[2 * nbin]);
              const cdf a0 = mul_conj(q0, la), a1 = mul_conj(q1, lb), b0 = mul_conj(q1, la), b1 = mul_conj(q2, lb);
              y = cdf{dfl_add(y.re, dfl_add(a0.re, a1.re)), dfl_add(y.im, dfl_add(a0.im, a1.im))};
              w = cdf{dfl_add(w.re, dfl_add(b0.re, b1.re)), dfl_add(w.im, dfl_add(b0.im, b1.im))};
            }
            hh = dfl_add(hh, dfl_add(re_mul(ra, y), re_mul(rb, w)));
          }
          v[c] += df_to(dh);
          v[3 + c] += df_to(hh);
        }
      }
    } else {
      for (int b = threadIdx.x < H.nt ? threadIdx.x : H.ne; b < H.ne - 1; b += H.nt) {
#pragma unroll 1
        for (int c = 0; c < 3; ++c) {
          double dh, hh;
          if (!XC || !het_bin_fx(H, b, c, rsh, dh, hh))
            het_bin_fp64(H, b, c, [&](int e, int md) { return rsh[(e * kNModes + md) * 3 + c]; }, dh, hh);
          v[c] += dh;
          v[3 + c] += hh;
        }
      }
    }
    het_block_sum(v, sh);
    if (threadIdx.x == 0) {
      for (int c = 0; c < 3; ++c) {
        L += v[c] - 0.5 * v[3 + c] - 0.5 * D.dd[c];
        if (dhhh) {
          dhhh[(((size_t)s * hs.n + I) * 3 + c) * 2 + 0] = v[c];
          dhhh[(((size_t)s * hs.n + I) * 3 + c) * 2 + 1] = v[3 + c];
        }
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) logl[s] = S.valid ? L : -INFINITY;
}

}  // namespace pe

// ------------------------------------------------------------------------------------------
// Host side
// ------------------------------------------------------------------------------------------
struct pe_hetero_s {
  pe::HetDev dev;
  void* mem;
  int device;
};

namespace {

constexpr double kMsunSh = 4.925490947641267e-6;
const double kGam[5] = {-5.0 / 3.0, -2.0 / 3.0, 1.0, 5.0 / 3.0, 7.0 / 3.0};
const int kModeMh[pe::kNModes] = {2, 1, 3, 2, 4};

double phase_metric(double f, double flo, double fhi) {
  double s = 0.0;
  for (double g : kGam) s += (g < 0 ? -1.0 : 1.0) * std::pow(f / (g < 0 ? flo : fhi), g);
  return s;
}
double fisco_of(const double* th) { return std::pow(6.0, -1.5) / (2.0 * pe::kPi * th[0] * kMsunSh); }

// Taper marks 1 - 0.1 * 0.7^j (j = 0..10) of m F_isco, as grid indices; kend: last bin below it.
void taper_marks(double T, long long k0, double fisco, int m, long long ks[11], long long* kend) {
  const double fe = m * fisco;
  for (int j = 0; j < 11; ++j) ks[j] = (long long)std::ceil((1.0 - 0.1 * std::pow(0.7, j)) * fe * T) - k0;
  *kend = (long long)std::ceil(fe * T) - k0 - 1;
}

bool mask_ok(unsigned m) { return (m & PE_MODE_ALL) != 0u && (m & ~(PE_MODE_ALL | PE_PREC_MIXED)) == 0u; }

pe_status herr(pe_status st, const char* msg) { return pe::set_error(st, msg); }

}  // namespace

extern "C" {

pe_status pe_hetero_default_edges(double T_obs, int64_t k0, int64_t nbins, const double* theta0, unsigned mode_mask,
                                  int nbins_coarse, int64_t* out_edges, int* inout_n) {
  if (theta0 == nullptr || out_edges == nullptr || inout_n == nullptr)
    return herr(PE_EINVAL, "pe_hetero_default_edges: NULL argument");
  if (!(T_obs > 0.0) || k0 < 1 || nbins < 2 || nbins_coarse < 1 || !mask_ok(mode_mask) || !(theta0[0] > 0.0))
    return herr(PE_EINVAL, "pe_hetero_default_edges: bad grid, mask, theta0 or bin count");
  const double fisco = fisco_of(theta0);
  double fend = 0.0;
  for (int md = 0; md < pe::kNModes; ++md)
    if ((mode_mask >> md) & 1u) fend = std::max(fend, kModeMh[md] * fisco);
  const long long kmax = std::min<long long>(nbins - 1, (long long)std::ceil(fend * T_obs) - k0 - 1);
  if (kmax < 1) return herr(PE_EINVAL, "pe_hetero_default_edges: the reference's band ends below the grid");
  const double flo = k0 / T_obs, fhi = (k0 + kmax) / T_obs;
  const double p0 = phase_metric(flo, flo, fhi), p1 = phase_metric(fhi, flo, fhi);
  std::set<long long> cand = {0, kmax};
  for (int j = 1; j < nbins_coarse; ++j) {
    const double target = p0 + (p1 - p0) * j / nbins_coarse;
    double a = flo, b = fhi;
    for (int it = 0; it < 200; ++it) {
      const double mid = 0.5 * (a + b);
      if (phase_metric(mid, flo, fhi) < target) a = mid; else b = mid;
    }
    cand.insert((long long)std::llround(0.5 * (a + b) * T_obs) - k0);
  }
  std::vector<std::pair<long long, long long>> forbid;   // (last mark, kend) per mode
  for (int md = 0; md < pe::kNModes; ++md) {
    if (!((mode_mask >> md) & 1u)) continue;
    long long ks[11], kend;
    taper_marks(T_obs, k0, fisco, kModeMh[md], ks, &kend);
    for (long long k : ks) cand.insert(k);
    forbid.push_back({ks[10], kend});
  }
  std::vector<int64_t> keep;
  for (long long k : cand) {
    if (k < 0 || k > kmax) continue;
    bool bad = false;
    if (k != kmax)
      for (auto& fb : forbid) bad |= (k > fb.first && k <= fb.second);
    if (!bad) keep.push_back(k);
  }
  if ((int)keep.size() > *inout_n) {
    char msg[160];
    snprintf(msg, sizeof(msg), "pe_hetero_default_edges: %zu edges do not fit in %d", keep.size(), *inout_n);
    return herr(PE_EINVAL, msg);
  }
  std::copy(keep.begin(), keep.end(), out_edges);
  *inout_n = (int)keep.size();
  return PE_OK;
}

pe_status pe_hetero_create(pe_detector det, const double* theta0, unsigned mode_mask, const int64_t* edges,
                           int nedges, pe_hetero* out) {
  if (out == nullptr || theta0 == nullptr || edges == nullptr) return herr(PE_EINVAL, "pe_hetero_create: NULL argument");
  *out = nullptr;
  if (!mask_ok(mode_mask)) return herr(PE_EINVAL, "pe_hetero_create: bad mode mask (PE_PREC_FP32 is not taken)");
  pe::DetSet ds;
  pe_status s0 = pe::detset_from_handles(&det, 1, &ds);
  if (s0 != PE_OK) return s0;
  const pe::DetDev& D = ds.d[0];
  const int ne = nedges;
  if (ne < 2 || ne > pe::kHetMaxEdges) return herr(PE_EINVAL, "pe_hetero_create: nedges outside [2, 640]");
  for (int i = 0; i < ne; ++i) {
    if (edges[i] < 0 || edges[i] >= D.nb || (i > 0 && edges[i] <= edges[i - 1]))
      return herr(PE_EINVAL, "pe_hetero_create: edges must increase strictly inside the grid");
  }
  for (int i = 0; i < PE_NPARAM; ++i)
    if (!std::isfinite(theta0[i])) return herr(PE_EINVAL, "pe_hetero_create: theta0 is not finite");
  const int K = (int)edges[ne - 1] + 1;
  const int nb = ne - 1;
  // one allocation: edge [ne] int, src [ne][5][3] int, fe [ne] double, h0e [ne][15], A [nb][30], Bs [nb][kPairs*9]
  auto a256 = [](size_t x) { return (x + 255) & ~size_t(255); };
  const size_t o_edge = 0;
  const size_t o_src = a256(o_edge + ne * sizeof(int));
  const size_t o_fe = a256(o_src + (size_t)ne * 15 * sizeof(int));
  const size_t o_h0e = a256(o_fe + ne * sizeof(double));
  const size_t o_A = a256(o_h0e + (size_t)ne * 15 * sizeof(double2));
  const size_t o_B = a256(o_A + (size_t)nb * 30 * sizeof(double2));
  const size_t o_Aw = a256(o_B + (size_t)nb * pe::kPairs * 9 * sizeof(double2));
  const size_t o_Bw = a256(o_Aw + (size_t)nb * 30 * sizeof(float4));
  const size_t o_Ax = a256(o_Bw + (size_t)nb * pe::kPairs * 9 * sizeof(float4));
  const size_t o_Bx = a256(o_Ax + (size_t)nb * 30 * sizeof(longlong2));
  const size_t o_Gx = a256(o_Bx + (size_t)nb * pe::kPairs * 9 * sizeof(longlong2));
  const size_t bytes = o_Gx + (size_t)nb * 3 * (pe::kNModes + 1) * sizeof(int);
  pe_hetero_s* h = new (std::nothrow) pe_hetero_s();
  if (!h) return herr(PE_ENOMEM, "pe_hetero_create: host allocation failed");
  cudaGetDevice(&h->device);
  if (pe::dmalloc(&h->mem, bytes) != cudaSuccess) {
    cudaGetLastError();
    delete h;
    return herr(PE_ENOMEM, "pe_hetero_create: device allocation failed");
  }
  unsigned char* base = static_cast<unsigned char*>(h->mem);
  int* d_edge = reinterpret_cast<int*>(base + o_edge);
  int* d_src = reinterpret_cast<int*>(base + o_src);
  double* d_fe = reinterpret_cast<double*>(base + o_fe);
  double2* d_h0e = reinterpret_cast<double2*>(base + o_h0e);
  double2* d_A = reinterpret_cast<double2*>(base + o_A);
  double2* d_B = reinterpret_cast<double2*>(base + o_B);
  float4* d_Aw = reinterpret_cast<float4*>(base + o_Aw);
  float4* d_Bw = reinterpret_cast<float4*>(base + o_Bw);
  longlong2* d_Ax = reinterpret_cast<longlong2*>(base + o_Ax);
  longlong2* d_Bx = reinterpret_cast<longlong2*>(base + o_Bx);
  int* d_Gx = reinterpret_cast<int*>(base + o_Gx);
  std::vector<int> he(ne);
  std::vector<double> hfe(ne);
  for (int i = 0; i < ne; ++i) {
    he[i] = (int)edges[i];
    hfe[i] = double(D.k0 + edges[i]) / D.T;
  }
  double* th0 = nullptr;
  pe::SampleCoef* coef = nullptr;
  int* nend = nullptr;
  double2* hb = nullptr;
  cudaError_t e = pe::dmalloc(&th0, PE_NPARAM * sizeof(double));
  if (e == cudaSuccess) e = pe::dmalloc(&coef, sizeof(pe::SampleCoef));
  if (e == cudaSuccess) e = pe::dmalloc(&nend, sizeof(int));
  if (e == cudaSuccess) e = pe::dmalloc(&hb, (size_t)pe::kNModes * 3 * K * sizeof(double2));
  if (e == cudaSuccess) e = pe::upload(th0, theta0, PE_NPARAM * sizeof(double));
  if (e == cudaSuccess) e = pe::upload(d_edge, he.data(), ne * sizeof(int));
  if (e == cudaSuccess) e = pe::upload(d_fe, hfe.data(), ne * sizeof(double));
  if (e == cudaSuccess) e = pe::launch_prep(th0, 1, mode_mask, ds, coef, nend, nullptr, 0);
  if (e == cudaSuccess) {
    auto kb = D.fx_ok ? pe::k_mode_brackets<true> : pe::k_mode_brackets<false>;
    kb<<<(K + pe::kTileBins - 1) / pe::kTileBins, pe::kTileBins>>>(D, coef, K, mode_mask, hb);
    e = pe::launch_status();
  }
  // reference brackets at the edges, and the carry-forward sources
  std::vector<double2> h0e((size_t)ne * 15);
  if (e == cudaSuccess) {
    pe::k_gather_edges<<<(ne * 15 + 127) / 128, 128>>>(hb, K, d_edge, ne, d_h0e);
    e = pe::launch_status();
  }
  if (e == cudaSuccess) e = cudaMemcpy(h0e.data(), d_h0e, h0e.size() * sizeof(double2), cudaMemcpyDeviceToHost);
  std::vector<int> src((size_t)ne * 15, -1);
  if (e == cudaSuccess) {
    const double fisco = fisco_of(theta0);
    for (int md = 0; md < pe::kNModes; ++md) {
      long long klast = -1;
      if ((mode_mask >> md) & 1u) {
        long long ks[11], kend;
        taper_marks(D.T, D.k0, fisco, kModeMh[md], ks, &kend);
        klast = ks[10];
      }
      for (int c = 0; c < 3; ++c)
        for (int i = 0; i < ne; ++i) {
          const size_t j = ((size_t)i * pe::kNModes + md) * 3 + c;
          const bool ok = he[i] <= klast && (h0e[j].x != 0.0 || h0e[j].y != 0.0);
          src[j] = ok ? i : (i > 0 ? src[j - 15] : -1);
        }
    }
    e = pe::upload(d_src, src.data(), src.size() * sizeof(int));
  }
  if (e == cudaSuccess) {   // the per-sample kernel multiplies by the inverses (no division per ratio)
    pe::k_invert_edges<<<(ne * 15 + 127) / 128, 128>>>(d_h0e, ne * 15);
    e = pe::launch_status();
  }
  if (e == cudaSuccess) {
    const long long n = (long long)nb * (30 + pe::kPairs * 9);
    pe::k_het_summary<<<(unsigned)((n + 127) / 128), 128>>>(D, d_edge, d_fe, ne, hb, K, d_A, d_B);
    e = pe::launch_status();
  }
  if (e == cudaSuccess) {   // double-word and fixed-point copies of the summary data
    pe::k_het_dw<<<(3 * nb + 127) / 128, 128>>>(d_fe, ne, d_A, d_B, d_Aw, d_Bw);
    pe::k_het_words<<<(3 * nb + 127) / 128, 128>>>(d_fe, ne, d_A, d_B, d_Ax, d_Bx, d_Gx);
    e = pe::launch_status();
  }
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  pe::dfree(th0);
  pe::dfree(coef);
  pe::dfree(nend);
  pe::dfree(hb);
  if (e != cudaSuccess) {
    cudaGetLastError();
    pe::dfree(h->mem);
    delete h;
    char msg[200];
    snprintf(msg, sizeof(msg), "pe_hetero_create: %s", cudaGetErrorString(e));
    return herr(PE_ECUDA, msg);
  }
  h->dev.det = D;
  h->dev.edge = d_edge;
  h->dev.fe = d_fe;
  h->dev.ih0e = d_h0e;
  h->dev.src = d_src;
  h->dev.A = d_A;
  h->dev.Bs = d_B;
  h->dev.Aw = d_Aw;
  h->dev.Bw = d_Bw;
  h->dev.Ax = d_Ax;
  h->dev.Bx = d_Bx;
  h->dev.Gx = d_Gx;
  h->dev.ne = ne;
  h->dev.nt = pe::het_threads(ne);
  h->dev.mask = mode_mask;
  *out = h;
  return PE_OK;
}

pe_status pe_hetero_destroy(pe_hetero h) {
  if (h == nullptr) return PE_OK;
  cudaDeviceSynchronize();
  pe::dfree(h->mem);
  cudaGetLastError();
  delete h;
  return PE_OK;
}

pe_status pe_hetero_loglike_batch(const pe_hetero* hets, int ndet, const double* theta, int B, double* out_logl,
                                  double* out_dhhh, int32_t* out_status, void* stream) {
  if (hets == nullptr || theta == nullptr || out_logl == nullptr) return herr(PE_EINVAL, "pe_hetero_loglike_batch: NULL");
  if (ndet < 1 || ndet > pe::kMaxDet) return herr(PE_EINVAL, "pe_hetero_loglike_batch: ndet outside [1, 8]");
  if (B < 1 || B > (1 << 20)) return herr(PE_EINVAL, "pe_hetero_loglike_batch: B outside [1, 2^20]");
  pe::HetSet hs;
  memset(&hs, 0, sizeof(hs));
  pe::DetSet ds;
  memset(&ds, 0, sizeof(ds));
  hs.n = ndet;
  ds.ndet = ndet;
  int dev = 0, nemax = 0;
  cudaGetDevice(&dev);
  for (int i = 0; i < ndet; ++i) {
    if (hets[i] == nullptr) return herr(PE_EINVAL, "pe_hetero_loglike_batch: NULL handle");
    if (hets[i]->device != dev) return herr(PE_EINVAL, "pe_hetero_loglike_batch: handle on another device");
    if (hets[i]->dev.mask != hets[0]->dev.mask) return herr(PE_EINVAL, "pe_hetero_loglike_batch: mode masks differ");
    hs.h[i] = hets[i]->dev;
    ds.d[i] = hets[i]->dev.det;
    nemax = std::max(nemax, hets[i]->dev.ne);
  }
  hs.nemax = nemax;
  auto is_dev = [](const void* p) {
    if (p == nullptr) return false;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) { cudaGetLastError(); return false; }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
  };
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  std::vector<void*> bufs;
  cudaError_t e = cudaSuccess;
  auto alloc = [&](void** p, size_t n) {
    if (e != cudaSuccess) return;
    e = pe::dmalloc_async(p, n + 16, st);
    if (e == cudaSuccess) bufs.push_back(*p);
  };
  const double* th = theta;
  if (!is_dev(theta)) {
    void* t = nullptr;
    alloc(&t, (size_t)B * PE_NPARAM * sizeof(double));
    if (e == cudaSuccess) e = pe::upload_async(t, theta, (size_t)B * PE_NPARAM * sizeof(double), st);
    th = static_cast<const double*>(t);
  }
  void *coef = nullptr, *nend = nullptr, *ll = out_logl, *dh = out_dhhh, *stt = out_status;
  alloc(&coef, (size_t)B * sizeof(pe::SampleCoef));
  alloc(&nend, (size_t)B * ndet * sizeof(int));
  const bool hl = !is_dev(out_logl), hd = out_dhhh && !is_dev(out_dhhh), hsx = out_status && !is_dev(out_status);
  if (hl) alloc(&ll, (size_t)B * sizeof(double));
  if (hd) alloc(&dh, (size_t)B * ndet * 6 * sizeof(double));
  if (hsx) alloc(&stt, (size_t)B * sizeof(int32_t));
  if (e == cudaSuccess)
    e = pe::launch_prep(th, B, hets[0]->dev.mask, ds, static_cast<pe::SampleCoef*>(coef), static_cast<int*>(nend),
                        static_cast<int*>(stt), st);
  const bool mix = (hets[0]->dev.mask & PE_PREC_MIXED) != 0u;
  const bool fxu = pe::fx_all_ok(ds);
  const size_t smem = (size_t)nemax * pe::kNModes * 3 * sizeof(double2) + (mix ? (size_t)nemax : 0);   // and the flags
  auto kern = mix ? (fxu ? pe::k_het_loglike<true, true> : pe::k_het_loglike<true, false>)
                  : (fxu ? pe::k_het_loglike<false, true> : pe::k_het_loglike<false, false>);
  int threads = 0;
  for (int i = 0; i < ndet; ++i) threads = std::max(threads, hs.h[i].nt);
  static_assert(pe::kProj <= 64, "one thread per form");
  if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) {
    kern<<<B, threads, smem, st>>>(hs, B, static_cast<const pe::SampleCoef*>(coef), static_cast<double*>(ll),
                                         static_cast<double*>(dh));
    e = pe::launch_status();
  }
  if (e == cudaSuccess && hl) e = cudaMemcpyAsync(out_logl, ll, (size_t)B * sizeof(double), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess && hd)
    e = cudaMemcpyAsync(out_dhhh, dh, (size_t)B * ndet * 6 * sizeof(double), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess && hsx) e = cudaMemcpyAsync(out_status, stt, (size_t)B * sizeof(int32_t), cudaMemcpyDeviceToHost, st);
  for (void* p : bufs) pe::dfree_async(p, st);
  if (e == cudaSuccess && (hl || hd || hsx)) e = pe::wait_stream(st);
  if (e == cudaErrorNotReady) return herr(PE_ETIMEOUT, "pe_hetero_loglike_batch: stream did not finish within the wait limit");
  if (e != cudaSuccess) {
    cudaGetLastError();
    char msg[200];
    snprintf(msg, sizeof(msg), "pe_hetero_loglike_batch: %s", cudaGetErrorString(e));
    return herr(PE_ECUDA, msg);
  }
  return PE_OK;
}

}  // extern "C"

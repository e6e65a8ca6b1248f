// pe_grad.cu -- kernels of the gradient (row G1) and Fisher matrix (row G2) of the Whittle
// log-likelihood (arXiv:2602.12011 Sec. 2.2 and the automatic-differentiation discussion of
// Sec. 2.3), built on the hand-written reverse sweep in pe_adjoint.cuh:
//   k_prep          per-sample coefficients and their derivatives in theta (pe_prep.cuh)
//   k_grad_fwd_tape FP64, persistent, two 128-thread CTAs per SM (mixed: three): per bin the forward mode sum
//                   writing each unit's tape (the CTA's region of global memory), the cotangents of the A/E/T
//                   sums dL/dB_c = conj(dg_c) - gg_c B_c, one reverse sweep per mode from the
//                   tape, and per tile the contraction of the form cotangents (pe_adjoint_tape.cuh)
//   k_grad_fwd_mixed the same in mixed precision with a double-word tape
//                   (pe_adjoint_tape_mixed.cuh)
//   k_grad_fwd_fx   both precisions where every detector takes the fixed-point unit, four CTAs per SM: the same with the
//                   sweeps in fixed point (pe_adjoint_fx.cuh); the two kernels above serve the other detectors
//   k_grad_reduce_warp, k_grad_reduce  fixed-order per-sample sums of the tile partials -> logL, grad[11], a warp per
//                   sample on small grids, a CTA on larger ones
//   k_fisher_fwd    per bin six reverse sweeps (Re/Im of X', Y', Z') by six warps -> Jacobian J, then
//                   F += sum_c gg_c (J_Re B_c^T J_Re B_c + J_Im B_c^T J_Im B_c)
//   k_fisher_fx     the same on the fixed-point unit: one forward pass per mode onto a tape in shared memory that six
//                   warps' sweeps (Re/Im of A', E', T') read
//   k_fisher_reduce fixed-order per-sample sums -> F[11][11]
#include <cuda_runtime.h>

#include "pe_adjoint.cuh"
#include "pe_adjoint_fx.cuh"
#include "pe_adjoint_mixed.cuh"
#include "pe_adjoint_tape.cuh"
#include "pe_adjoint_tape_mixed.cuh"
#include "pe_grad.h"
#include "pe_kernels.h"
#include "pe_fault.h"
#include "pe_prep.cuh"

namespace pe {

constexpr int kGradW = 23;   // per-tile partials: dh[3], hh[3], M q c1 c2 dL io ph tc, k[3] p[3] q[3]
constexpr int kGradV = 14;   // of which reduced by shuffles: dh[3], hh[3], M q c1 c2 dL io ph tc
constexpr int kFisherW = 66; // unique entries of the symmetric 11 x 11 matrix

__device__ __forceinline__ int find_pair_g(const long long* off, int P, long long t) {
  int lo = 0, hi = P;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (off[mid] <= t) lo = mid; else hi = mid;
  }
  return lo;
}

// Cotangents of the A/E/T sums of one bin, and the bin's likelihood terms:
//   L_c = Re(dg_c B_c) - gg_c |B_c|^2 / 2  =>  Bbar_c = (dg.x - gg B.x, -dg.y - gg B.y).
// (The brackets' cotangents follow from B_A = Z' - X', B_E = X' - 2Y' + Z', B_T = X' + Y' + Z';
// link_seeds forms what the link sweeps need from them.)
__device__ __forceinline__ void aet_cotangents(const DetDev& D, int b, const double2 o[3], double v6[6],
                                               double2 bb[3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double2 g = D.dg[c * D.nb + b];
    const double w = D.gg[c * D.nb + b];
    v6[c] += g.x * o[c].x - g.y * o[c].y;
    v6[3 + c] += w * (o[c].x * o[c].x + o[c].y * o[c].y);
    bb[c] = make_double2(g.x - w * o[c].x, -g.y - w * o[c].y);
  }
}

// Block sum of the kGradV per-thread partials, already stored in red[i][threadIdx.x], through
// shared memory in a fixed order (block_sum6's scheme for 14 rows): thread t < 112 adds entries
// g, g + 8, ..., g + 120 of row i = t / 8 (g = t % 8) into red[i][g]; thread i < 14 then adds
// red[i][0..7] and returns the row's sum (other threads return 0). About 1,800 FP64 additions per
// tile against ~9,000 for a shuffle tree over all lanes. The caller stores the partials and holds
// the barrier before them.
__device__ __forceinline__ double grad_block_sum(double (*red)[kTileBins + kRedPad]) {
  __syncthreads();
  if (threadIdx.x < kGradV * 8) {
    const int i = threadIdx.x >> 3, g = threadIdx.x & 7;
    double s = red[i][g];
#pragma unroll
    for (int k = 1; k < kTileBins / 8; ++k) s += red[i][g + 8 * k];
    red[i][g] = s;   // only this thread touches column g of row i in this step
  }
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x < kGradV) {
    s = red[threadIdx.x][0];
#pragma unroll
    for (int g = 1; g < 8; ++g) s += red[threadIdx.x][g];
  }
  return s;
}

// Mixed-precision gradient with a double-word tape (pe_adjoint_tape_mixed.cuh): per tile the
// mixed-precision forward mode sum writes each unit's tape, the bracket cotangents are formed in
// FP64 from the mode sum, the reverse sweeps read the tape and run in double words (their theta
// components return to FP64 once per bin), and the CTA contracts the form cotangents in double
// words. The 23 partials per tile are the FP64 kernel's.
__global__ void __launch_bounds__(kTileBins, 3) k_grad_fwd_mixed(DetSet ds, int B, const SampleCoef* __restrict__ coef,
                                                              const SampleGrad* __restrict__ sgrad,
                                                              const int* __restrict__ nend,
                                                              const long long* __restrict__ off, double* part,
                                                              double* tape_all) {
  df* tape = reinterpret_cast<df*>(tape_all + (size_t)blockIdx.x * kTapeDoubles);
  __shared__ double red[kGradV][kTileBins + kRedPad];
  __shared__ unsigned tile_used;   // the slots some unit of the tile used
  __shared__ float4 stabw[kSinTab];
  __shared__ cdf lseed[6][kTileBins];   // each thread's link seeds P_l, Q_l (own column)
  __shared__ ChainW cw;                  // the tile's chain-rule coefficients as double words
  __shared__ double pc[kProj];
  __shared__ float2 pcw[kProj];
  __shared__ double sums[3][kTapeSums];
  for (int i = threadIdx.x; i < kSinTab; i += blockDim.x) stabw[i] = ds.d[0].sctw[i];
  __syncthreads();
  const int P = ds.ndet * B;
  const long long total = off[P];
  df* tcol = tape + threadIdx.x;
  const unsigned long long pol = tape_l2_policy();
  for (long long t = blockIdx.x; t < total; t += gridDim.x) {
    const int p = find_pair_g(off, P, t);
    if (!PE_CHK(p >= 0 && p < P && off[p + 1] <= total && nend[p] <= ds.d[p / B].nb, 16)) continue;
    const int I = p / B, s = p - I * B;
    const int b = int(t - off[p]) * kTileBins + threadIdx.x;
    const DetDev& D = ds.d[I];
    if (threadIdx.x == 0) tile_used = 0u;   // the previous tile's readers passed two barriers since
    proj_prologue(D, coef[s], pc);
    if (threadIdx.x < kProj) pcw[threadIdx.x] = to_dw(pc[threadIdx.x]);
    chain_fill(D, coef[s], sgrad[s], &cw);
    __syncthreads();
    double v[kGradV];
#pragma unroll
    for (int i = 0; i < kGradV; ++i) v[i] = 0.0;
    unsigned used = 0;
    if (b < nend[p]) {
      const SampleCoef& S = coef[s];
      const SampleGrad& SG = sgrad[s];
      BinIn Bn;
      load_bin(D, b, S.tc, Bn);
      BinW W;
      load_bin_w(D, b, W);
      const float4 zz = D.zw[b];
      const cdf zw = {df_make(zz.x, zz.y), df_make(zz.z, zz.w)};
      MixAcc xa;
      mix_zero(xa);
#pragma unroll 1
      for (int md = 0; md < kNModes; ++md) {
        if (md == 3 && S.pair32) continue;
        const ModeCoef& C = S.md[md];
        if (!C.active || !dlt_pos(Bn.f, C.fend)) continue;
        const int sl = tape_slot(md);
        mode_fwd_tape_mixed(D, S, C, Bn, W, xa, stabw, pcw, (md == 0 && S.pair32) ? &S.md[3] : nullptr,
                            tcol + sl * kTapeF * kTileBins, pol);
        used |= 1u << sl;
      }
      cdf x[3], od[3];
      mix_final(xa, zw, x);
      aet_from_xyz_dw(x, od);
      double2 o[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) o[c] = make_double2(df_to(od[c].re) * S.ihsc, df_to(od[c].im) * S.ihsc);
      double2 bb[3];
      aet_cotangents(D, b, o, v, bb);
      const double ih = S.ihsc;
      cdf bw[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) bw[c] = cdf{df_from_bits(bb[c].x * ih), df_from_bits(bb[c].y * ih)};
      link_seeds_dw(bw, W.sa, W.ca, &lseed[0][threadIdx.x]);
      const df lnf3 = df_from_bits(Bn.lnf3);
      GradAcc g;
      gacc_zero(g);
      GradAccDW gw;
      gaccdw_zero(gw);
#pragma unroll 1
      for (int md = 0; md < kNModes; ++md) {
        if (md == 3 && S.pair32) continue;
        const ModeCoef& C = S.md[md];
        if (!C.active || !dlt_pos(Bn.f, C.fend)) continue;
        mode_bwd_tape_mixed(D, S, SG, md, Bn, W, &lseed[0][threadIdx.x], cw, lnf3, gw, g, pcw,
                            tcol + tape_slot(md) * kTapeF * kTileBins, (md == 0 && S.pair32) ? 3 : -1, pol);
      }
      gaccdw_flush(gw, g);
      v[6] = g.M; v[7] = g.q; v[8] = g.c1; v[9] = g.c2; v[10] = g.dL; v[11] = g.io; v[12] = g.ph; v[13] = g.tc;
    }
#pragma unroll 1
    for (int sl = 0; sl < kTapeSlots; ++sl)
      if (!(used & (1u << sl))) tape_clear_dw(tcol + sl * kTapeF * kTileBins, pol);
    {
      const unsigned wu = __reduce_or_sync(0xffffffffu, used);
      if ((threadIdx.x & 31) == 0 && wu) atomicOr(&tile_used, wu);
    }
    __syncthreads();   // the tape is complete; the previous tile's readers of red are done
#pragma unroll
    for (int i = 0; i < kGradV; ++i) red[i][threadIdx.x] = v[i];
    // the contraction walks only the slots some unit of the tile used
    const unsigned tu = tile_used;
    unsigned act = 0;
    int nact = 0;
#pragma unroll
    for (int sl = 0; sl < kTapeSlots; ++sl)
      if ((tu >> sl) & 1u) act |= unsigned(sl) << (2 * nact++);
    const int ent = nact * kTileBins;
    if (threadIdx.x < 3 * kTapeSums) {
      const int j = threadIdx.x % kTapeSums, q = threadIdx.x / kTapeSums;
      const int e0 = q * ent / 3, e1 = (q + 1) * ent / 3;
      sums[q][j] = tape_sum_dw(tape, j, e0, e1, D.orbit != 0, act, pol);
    }
    const double a = grad_block_sum(red);
    if (threadIdx.x < kGradV) {
      part[t * kGradW + threadIdx.x] = a;
    } else if (threadIdx.x < kGradW) {
      const int k = threadIdx.x - kGradV;
      double pcb[kTapeSums];
      for (int j = 0; j < kTapeSums; ++j) pcb[j] = sums[0][j] + sums[1][j] + sums[2][j];
      part[t * kGradW + threadIdx.x] = tape_to_frame(D, pcb, k / 3, k % 3);
    }
  }
}

// FP64 gradient with a tape. Per tile: the forward mode sum writes each unit's tape, the bracket
// cotangents follow from the mode sum, the reverse sweeps read the tape and leave the form
// cotangents in it, and the CTA contracts them with the orbit basis (42 sums over the tile's
// 512 (bin, slot) entries, three threads per sum) and maps the sums to the sky frame. The 23
// partials per tile are those of the recomputing kernel.
__global__ void __launch_bounds__(kTileBins, 2) k_grad_fwd_tape(DetSet ds, int B, const SampleCoef* __restrict__ coef,
                                                             const SampleGrad* __restrict__ sgrad,
                                                             const int* __restrict__ nend,
                                                             const long long* __restrict__ off, double* part,
                                                             double* tape_all) {
  double* tape = tape_all + (size_t)blockIdx.x * kTapeDoubles;   // [kTapeSlots][kTapeF][kTileBins]
  __shared__ double red[kGradV][kTileBins + kRedPad];
  __shared__ unsigned tile_used;   // the slots some unit of the tile used
  __shared__ double2 stab[kSinTab];
  __shared__ double2 lseed[6][kTileBins];   // each thread's link seeds P_l, Q_l (own column)
  __shared__ double pc[kProj];
  __shared__ double sums[3][kTapeSums];
  for (int i = threadIdx.x; i < kSinTab; i += blockDim.x) stab[i] = ds.d[0].sct[i];
  __syncthreads();
  const int P = ds.ndet * B;
  const long long total = off[P];
  double* tcol = tape + threadIdx.x;
  const unsigned long long pol = tape_l2_policy();
  for (long long t = blockIdx.x; t < total; t += gridDim.x) {
    const int p = find_pair_g(off, P, t);
    if (!PE_CHK(p >= 0 && p < P && off[p + 1] <= total && nend[p] <= ds.d[p / B].nb, 16)) continue;
    const int I = p / B, s = p - I * B;
    const int b = int(t - off[p]) * kTileBins + threadIdx.x;
    const DetDev& D = ds.d[I];
    if (threadIdx.x == 0) tile_used = 0u;   // the previous tile's readers passed two barriers since
    proj_prologue(D, coef[s], pc);
    double v[kGradV];
#pragma unroll
    for (int i = 0; i < kGradV; ++i) v[i] = 0.0;
    unsigned used = 0;
    if (b < nend[p]) {
      const SampleCoef& S = coef[s];
      const SampleGrad& SG = sgrad[s];
      BinIn Bn;
      load_bin(D, b, S.tc, Bn);
      XYZAcc xa;
      xyz_zero(xa);
#pragma unroll 1
      for (int md = 0; md < kNModes; ++md) {
        if (md == 3 && S.pair32) continue;
        const ModeCoef& C = S.md[md];
        if (!C.active || !dlt_pos(Bn.f, C.fend)) continue;
        const int sl = tape_slot(md);
        mode_fwd_tape(D, S, C, Bn, xa, stab, pc, (md == 0 && S.pair32) ? &S.md[3] : nullptr,
                      tcol + sl * kTapeF * kTileBins, pol);
        used |= 1u << sl;
      }
      double2 x[3], o[3];
      xyz_final(xa, Bn.z, x);
      aet_from_xyz(x, o);
      double2 bb[3];
      aet_cotangents(D, b, o, v, bb);
      link_seeds(bb, Bn.sa, Bn.ca, &lseed[0][threadIdx.x]);
      GradAcc g;
      gacc_zero(g);
#pragma unroll 1
      for (int md = 0; md < kNModes; ++md) {
        if (md == 3 && S.pair32) continue;
        const ModeCoef& C = S.md[md];
        if (!C.active || !dlt_pos(Bn.f, C.fend)) continue;
        mode_bwd_tape(D, S, SG, md, Bn, &lseed[0][threadIdx.x], g, pc,
                      tcol + tape_slot(md) * kTapeF * kTileBins, (md == 0 && S.pair32) ? 3 : -1, pol);
      }
      v[6] = g.M; v[7] = g.q; v[8] = g.c1; v[9] = g.c2; v[10] = g.dL; v[11] = g.io; v[12] = g.ph; v[13] = g.tc;
    }
#pragma unroll 1
    for (int sl = 0; sl < kTapeSlots; ++sl)
      if (!(used & (1u << sl))) tape_clear(tcol + sl * kTapeF * kTileBins, pol);
    {
      const unsigned wu = __reduce_or_sync(0xffffffffu, used);
      if ((threadIdx.x & 31) == 0 && wu) atomicOr(&tile_used, wu);
    }
    __syncthreads();   // the tape is complete; the previous tile's readers of red are done
#pragma unroll
    for (int i = 0; i < kGradV; ++i) red[i][threadIdx.x] = v[i];
    // the contraction walks only the slots some unit of the tile used
    const unsigned tu = tile_used;
    unsigned act = 0;
    int nact = 0;
#pragma unroll
    for (int sl = 0; sl < kTapeSlots; ++sl)
      if ((tu >> sl) & 1u) act |= unsigned(sl) << (2 * nact++);
    const int ent = nact * kTileBins;
    if (threadIdx.x < 3 * kTapeSums) {
      const int j = threadIdx.x % kTapeSums, q = threadIdx.x / kTapeSums;
      const int e0 = q * ent / 3, e1 = (q + 1) * ent / 3;
      sums[q][j] = tape_sum(tape, j, e0, e1, D.orbit != 0, act, pol);
    }
    const double a = grad_block_sum(red);
    if (threadIdx.x < kGradV) {
      part[t * kGradW + threadIdx.x] = a;
    } else if (threadIdx.x < kGradW) {
      const int k = threadIdx.x - kGradV;
      double pcb[kTapeSums];
      for (int j = 0; j < kTapeSums; ++j) pcb[j] = sums[0][j] + sums[1][j] + sums[2][j];
      part[t * kGradW + threadIdx.x] = tape_to_frame(D, pcb, k / 3, k % 3);
    }
  }
}

// The gradient on detectors that take the fixed-point unit, both precisions: per bin the forward mode sum writes each unit's
// tape, the A/E/T cotangents and link seeds follow in FP64, and the reverse sweeps run in fixed point from the tape
// (pe_adjoint_fx.cuh). Per tile 17 sums: the 14 of the FP64 kernel and the frame's three rotation cotangents, written as
// the 23 partials the reduction reads. Bound by the FP64 pipe (141 operations a unit, 67 % busy of 84 %) and dependent integer operations (5,600 thread
// instructions a unit). 64 LISA samples of 2^22 s: FP64 4.08 -> 1.54 ms; 500 at the mixed precision, whose
// double-word sweep was at the FP32 pipe's rate, 12.8 -> 10.8 ms; hence both precisions take it. (Items drawn from a counter and the
// bin's sums in shared memory: 1.34 and 9.9 ms; five and six CTAs per SM spill, 4 and 6 % slower.)
constexpr int kGradFxV = 17;
constexpr int kGradFxRows = 6 + kGSums;
constexpr int kGradFxCtas = 4;   // resident CTAs per SM (tape 92 MB, inside L2)
constexpr int kGradFxRow = 7;    // threads that add one row of the block sum
__global__ void __launch_bounds__(kTileBins, kGradFxCtas) k_grad_fwd_fx(DetSet ds, int B, const SampleCoef* __restrict__ coef,
                                                                      const SampleGrad* __restrict__ sgrad,
                                                                      const int* __restrict__ nend,
                                                                      const long long* __restrict__ off, double* part,
                                                                      double* tape_all, unsigned long long* ctr) {
  __shared__ long long next;
  __shared__ double red[kGradFxRows][kTileBins + kRedPad];   // the values of the block sums; before, from row 6 on, the bin's sums
  __shared__ fx col[kFxSums][kTileBins];   // the forward sums, then the link seeds, a column per thread
  __shared__ __align__(16) fx pc[kFxProjAll];
  __shared__ double rot[3];
  static_assert(kGradFxV * kGradFxRow <= kTileBins, "one pass adds every row");
  double* tape = tape_all + (size_t)blockIdx.x * kTapeDoubles + threadIdx.x;
  const int P = ds.ndet * B;
  const long long total = off[P];
  const unsigned long long pol = tape_l2_policy();
  for (long long t = blockIdx.x, tn = 0; t < total; t = work_next(tn, &next)) {
    tn = work_fetch(ctr, t);
    const int p = find_pair_warp(off, P, t);
    if (!PE_CHK(p >= 0 && p < P && off[p + 1] <= total && nend[p] <= ds.d[p / B].nb, 16)) continue;
    const int I = p / B, s = p - I * B;
    const int b = int(t - off[p]) * kTileBins + threadIdx.x;
    const DetDev& D = ds.d[I];
    const SampleCoef& S = coef[s];
    fx_proj_prologue(D, S, pc);   // its first barrier: the previous tile's readers of red and rot are done
    fx_proj3(pc);
    if (b < nend[p]) {
      const SampleGrad& SG = sgrad[s];
      FxBin Bn;
      load_bin_fx(D, b, S.tc, Bn);
      FxAcc a;
      fx_zero(a, &col[0][threadIdx.x]);
#pragma unroll 1
      for (int md = 0; md < kNModes; ++md) {
        if (md == 3 && S.pair32) continue;
        const ModeCoef& C = S.md[md];
        if (!C.active || !dlt_pos(Bn.f, C.fend)) continue;
        const FxTape tp = {tape + tape_slot(md) * kTapeF * kTileBins, pol};
        mode_bin_fx(D, S, C, Bn, a, ds.d[0].fcis, ds.d[0].fsinc, pc, md, (md == 0 && S.pair32) ? &S.md[3] : nullptr, tp);
      }
      double2 o[3], bb[3], pq[6];
      aet_from_fx(a, D.z[b], o);
      double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
      aet_cotangents(D, b, o, v, bb);
#pragma unroll
      for (int i = 0; i < 6; ++i) red[i][threadIdx.x] = v[i];
      const double2 sc = D.sca[b];
      link_seeds<1>(bb, sc.x, sc.y, pq);
      const int Es = fx_seeds<kTileBins>(pq, &col[0][threadIdx.x]);
      const fx a3 = fx_times_k((unsigned)(D.k0 + b), D.fx_a3);
      const double fm13 = D.fm13[b], invf = fm13 * fm13 * fm13, n2pif = -2.0 * kPi * Bn.f, fR = -D.R * n2pif;
      FxBinAccShared<kTileBins + kRedPad> ga = {&red[6][threadIdx.x]};
      ga.zero();
#pragma unroll 1
      for (int md = 0; md < kNModes; ++md) {
        if (md == 3 && S.pair32) continue;
        const ModeCoef& C = S.md[md];
        if (Es == 0 || Es == 0x7ff || !C.active || !dlt_pos(Bn.f, C.fend)) continue;
        const FxTape tp = {tape + tape_slot(md) * kTapeF * kTileBins, pol};
        mode_bwd_fx<kTileBins>(D, S, SG, md, (md == 0 && S.pair32) ? 3 : -1, Bn, fm13, invf, fR, n2pif, a3, &col[0][threadIdx.x], Es, ga, pc,
                               tp);
      }
      GradAcc g;
      fx_bin_grad(S, SG, ga, g);
      const double out[kGradFxV - 6] = {g.M, g.q, g.c1, g.c2, g.dL, g.io, g.ph, g.tc, g.k[0], g.k[1], g.k[2]};
#pragma unroll
      for (int i = 6; i < kGradFxV; ++i) red[i][threadIdx.x] = Es == 0x7ff ? __longlong_as_double(0x7ff8000000000000LL) : out[i - 6];   // seeds of inf or NaN data
    } else {
#pragma unroll
      for (int i = 0; i < kGradFxV; ++i) red[i][threadIdx.x] = 0.0;
    }
    __syncthreads();
    // thread t adds entries g, g + 7, ... of row i = t / 7 (g = t % 7) into red[i][g]; then thread i its seven
    if (threadIdx.x < kGradFxV * kGradFxRow) {
      const int i = threadIdx.x / kGradFxRow, g = threadIdx.x % kGradFxRow;
      double x = red[i][g];
      for (int k = g + kGradFxRow; k < kTileBins; k += kGradFxRow) x += red[i][k];
      red[i][g] = x;   // only this thread touches column g of row i in this step
    }
    __syncthreads();
    if (threadIdx.x < kGradFxV) {
      double x = red[threadIdx.x][0];
#pragma unroll
      for (int g = 1; g < kGradFxRow; ++g) x += red[threadIdx.x][g];
      if (threadIdx.x < kGradV) part[t * kGradW + threadIdx.x] = x;
      else rot[threadIdx.x - kGradV] = x;
    }
    __syncthreads();
    if (threadIdx.x >= kGradV && threadIdx.x < kGradW) {
      const int k = threadIdx.x - kGradV;
      part[t * kGradW + threadIdx.x] = rotation_to_frame(S, rot, k / 3, k % 3);
    }
  }
  work_done(ctr);
}

// logL and the gradient from the per-component sums over every detector's tiles.
__device__ __forceinline__ void grad_write(int s, double L, const double acc[kGradW], const SampleCoef* coef,
                                           const SampleGrad* sgrad, double* logl, double* grad) {
  const bool valid = coef[s].valid != 0;
  if (logl) logl[s] = valid ? L : -INFINITY;
  GradAcc g;
  g.M = acc[6]; g.q = acc[7]; g.c1 = acc[8]; g.c2 = acc[9]; g.dL = acc[10]; g.io = acc[11]; g.ph = acc[12];
  g.tc = acc[13];
  for (int i = 0; i < 3; ++i) { g.k[i] = acc[14 + i]; g.p[i] = acc[17 + i]; g.qv[i] = acc[20 + i]; }
  double out[PE_NPARAM];
  gacc_to_theta(g, sgrad[s], out);
  for (int i = 0; i < PE_NPARAM; ++i) grad[(size_t)s * PE_NPARAM + i] = valid ? out[i] : 0.0;
}

// Small grids (at most kGradWarpTiles tiles a detector): one warp per sample, fixed-order sums over each detector's tiles. (Whole calls,
// one warp and one CTA per sample: 8 tiles 87 and 86 us for one sample, 703 and 721 for 1024; 64 tiles 90 and 86, 5028 and 5053; 820 tiles
// 197 and 176 us for one sample, 7108 and 7082 for 128.)
constexpr int kGradWarpTiles = 64;
__global__ void k_grad_reduce_warp(DetSet ds, int B, const long long* off, const double* part, const SampleCoef* coef,
                              const SampleGrad* sgrad, double* logl, double* grad) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (warp >= B) return;
  const int s = warp;
  double acc[kGradW];
  for (int i = 0; i < kGradW; ++i) acc[i] = 0.0;
  double L = 0.0;
  for (int I = 0; I < ds.ndet; ++I) {
    const int p = I * B + s;
    if (!PE_CHK(off[p] >= 0 && off[p + 1] <= off[ds.ndet * B], 32)) continue;
    double v[kGradW];
    for (int i = 0; i < kGradW; ++i) v[i] = 0.0;
    for (long long t = off[p] + lane; t < off[p + 1]; t += 32)
      for (int i = 0; i < kGradW; ++i) v[i] += part[t * kGradW + i];
    for (int i = 0; i < kGradW; ++i)
      for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_down_sync(0xffffffffu, v[i], o);
    if (lane == 0) {
      for (int c = 0; c < 3; ++c) L += v[c] - 0.5 * v[3 + c] - 0.5 * ds.d[I].dd[c];
      for (int i = 6; i < kGradW; ++i) acc[i] += v[i];
    }
  }
  if (lane == 0) grad_write(s, L, acc, coef, sgrad, logl, grad);
}
// Larger grids: one CTA per sample, thread (r, i) adds component i of the tiles r, r + 32, ... (coalesced, four loads in flight),
// warp i adds the 32 rows (64 samples, LISA 2^22 s: 83 us with one warp per sample).
__global__ void __launch_bounds__(kGradW * 32) k_grad_reduce(DetSet ds, int B, const long long* off, const double* part,
                                                             const SampleCoef* coef, const SampleGrad* sgrad,
                                                             double* logl, double* grad) {
  __shared__ double red[kGradW][33];
  __shared__ double v[kGradW];
  const int s = blockIdx.x, i = threadIdx.x % kGradW, r = threadIdx.x / kGradW;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double acc[kGradW];
  for (int k = 0; k < kGradW; ++k) acc[k] = 0.0;
  double L = 0.0;
  for (int I = 0; I < ds.ndet; ++I) {
    const int p = I * B + s;
    long long t0 = off[p], t1 = off[p + 1];
    if (!PE_CHK(t0 >= 0 && t1 <= off[ds.ndet * B], 32)) t0 = t1;
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    for (long long t = t0 + r; t < t1; t += 128) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (t + 32 * k < t1) a[k] += part[(t + 32 * k) * kGradW + i];
    }
    red[i][r] = (a[0] + a[1]) + (a[2] + a[3]);
    __syncthreads();
    double x = red[w][lane];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if (lane == 0) v[w] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int c = 0; c < 3; ++c) L += v[c] - 0.5 * v[3 + c] - 0.5 * ds.d[I].dd[c];
      for (int k = 6; k < kGradW; ++k) acc[k] += v[k];
    }
  }
  if (threadIdx.x == 0) grad_write(s, L, acc, coef, sgrad, logl, grad);
}

// Fisher: six warps per 128-bin tile, in four 32-bin passes. Per pass warp j runs the reverse sweeps of seed j (Re/Im of X',
// Y', Z') over its lanes' bins, giving row j of the Jacobian; the warps then form the six A/E/T rows and each
// accumulates eleven of the 66 entries. A few points give a few hundred tiles: with one warp per tile, three warps
// an SM each ran 24 dependent sweeps of every mode (3.1 ms for three points on LISA, 2^21 s; 1.5 ms now, 1.7 at two CTAs per SM, whose 168 registers spill).
constexpr int kFisherWarps = 6;
__global__ void __launch_bounds__(32 * kFisherWarps, 1) k_fisher_fwd(DetSet ds, int B, const SampleCoef* __restrict__ coef,
                                                                    const SampleGrad* __restrict__ sgrad,
                                                                    const int* __restrict__ nend,
                                                                    const long long* __restrict__ off, double* part) {
  __shared__ double Js[kFisherWarps][PE_NPARAM][32];   // rows 0 Re X', 1 Im X', 2 Re Y', 3 Im Y', 4 Re Z', 5 Im Z'
  __shared__ double Ja[kFisherWarps][PE_NPARAM][32];   // rows Re/Im of B_A, B_E, B_T
  const int P = ds.ndet * B;
  const long long total = off[P];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (long long t = blockIdx.x; t < total; t += gridDim.x) {
    const int p = find_pair_g(off, P, t);
    if (!PE_CHK(p >= 0 && p < P && off[p + 1] <= total && nend[p] <= ds.d[p / B].nb, 64)) continue;
    const int I = p / B, s = p - I * B;
    const DetDev& D = ds.d[I];
    const SampleCoef& S = coef[s];
    const SampleGrad& SG = sgrad[s];
    double F[kFisherW / kFisherWarps];
#pragma unroll
    for (int e = 0; e < kFisherW / kFisherWarps; ++e) F[e] = 0.0;
#pragma unroll 1
    for (int sub = 0; sub < kTileBins / 32; ++sub) {
      const int b = int(t - off[p]) * kTileBins + sub * 32 + lane;
      const bool on = b < nend[p];
      double row[PE_NPARAM];
      if (on) {
        BinIn Bn;
        load_bin(D, b, S.tc, Bn);
        const double2 one = make_double2((w & 1) ? 0.0 : 1.0, (w & 1) ? 1.0 : 0.0);
        const double2 zero = make_double2(0.0, 0.0);
        GradAcc g;
        gacc_zero(g);
#pragma unroll 1
        for (int md = 0; md < kNModes; ++md) {
          if (md == 3 && S.pair32) continue;
          if (S.md[md].active && dlt_pos(Bn.f, S.md[md].fend))
            mode_bwd(D, S, SG, md, Bn, w / 2 == 0 ? one : zero, w / 2 == 1 ? one : zero, w / 2 == 2 ? one : zero, g, D.sct,
                     (md == 0 && S.pair32) ? 3 : -1);
        }
        gacc_to_theta(g, SG, row);
      } else {
#pragma unroll
        for (int i = 0; i < PE_NPARAM; ++i) row[i] = 0.0;
      }
#pragma unroll
      for (int i = 0; i < PE_NPARAM; ++i) Js[w][i][lane] = row[i];
      __syncthreads();
      const int c = w >> 1, ri = w & 1;
#pragma unroll
      for (int i = 0; i < PE_NPARAM; ++i) {
        const double X = Js[ri][i][lane], Y = Js[2 + ri][i][lane], Z = Js[4 + ri][i][lane];
        Ja[w][i][lane] = (c == 0) ? (Z - X) : (c == 1) ? (X - 2.0 * Y + Z) : (X + Y + Z);
      }
      __syncthreads();   // the next pass writes Js and, past its barrier, Ja
      // entries e = w, w + 6, ... of the upper triangle, row by row
#pragma unroll 1
      for (int r = 0; r < kFisherWarps; ++r) {
        const double g = on ? D.gg[(r >> 1) * D.nb + b] : 0.0;
        int i = 0, k = w;
        while (k >= PE_NPARAM - i) { k -= PE_NPARAM - i; ++i; }
#pragma unroll
        for (int e = 0; e < kFisherW / kFisherWarps; ++e) {
          F[e] = fma(g * Ja[r][i][lane], Ja[r][i + k][lane], F[e]);
          k += kFisherWarps;
          while (i < PE_NPARAM && k >= PE_NPARAM - i) { k -= PE_NPARAM - i; ++i; }
        }
      }
    }
    // fixed-order sums over the lanes
#pragma unroll
    for (int e = 0; e < kFisherW / kFisherWarps; ++e) {
      for (int o = 16; o > 0; o >>= 1) F[e] += __shfl_down_sync(0xffffffffu, F[e], o);
      if (lane == 0) part[t * kFisherW + w + kFisherWarps * e] = F[e];
    }
  }
}

// Sums over the lanes of the eleven values of each lane: in five steps a lane keeps half of its values, sends the
// other half and adds what it gets, 13 additions where eleven shuffle trees make 55. Lane l ends with the sum of value fisher_lane_entry(l)
// (-1: with none).
__host__ __device__ constexpr int fisher_kept(int step) { return step == 0 ? 6 : (step == 1 ? 3 : (step == 2 ? 2 : 1)); }   // of 11, 6, 3, 2, 1
static_assert(kFisherW / kFisherWarps == 11, "fisher_kept halves eleven values");
__device__ __forceinline__ double fisher_lane_sum(double v[kFisherW / kFisherWarps], int lane) {
#pragma unroll
  for (int st = 0; st < 5; ++st) {
    const int o = 16 >> st, keep = fisher_kept(st), have = st == 0 ? kFisherW / kFisherWarps : fisher_kept(st - 1);
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int k = 0; k < keep; ++k) {
      const double lo = v[k], hi = k + keep < have ? v[k + keep] : 0.0;
      v[k] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, o);
    }
  }
  return v[0];
}
__device__ __forceinline__ int fisher_lane_entry(int lane) {
  int first = 0, n = kFisherW / kFisherWarps;
#pragma unroll
  for (int st = 0; st < 5; ++st) {
    if (lane & (16 >> st)) {
      first += fisher_kept(st);
      n -= fisher_kept(st);
    } else {
      n = min(n, fisher_kept(st));
    }
  }
  return n > 0 ? first : -1;
}

// Fisher on detectors that take the fixed-point unit: six warps per 32 bins. Warps 0-3 first run the forward pass of one mode
// each (slot w) onto a tape in shared memory, with the chain factors that the seeds share; then warp j runs seed j's reverse
// sweeps (Re/Im of A', E', T'), giving row j of the Jacobian, and each warp accumulates eleven of the 66 entries. Bound by
// the dependent integer operations of the sweeps at 12 warps an SM and, at about 2,100 per bin, by the FP64 pipe.
// Three points on LISA, 2^21 s: 1.60 ms with the FP64 sweeps (k_fisher_fwd), 0.39 ms now.
constexpr int kFisherFxThreads = 32 * kFisherWarps;
struct FisherTape {   // field f of a lane at p[32 f]
  static constexpr bool kOn = true, kChain = true;
  fx* p;
  __device__ __forceinline__ void st(int f, fx v) const { p[f * 32] = v; }
  __device__ __forceinline__ fx ld(int f) const { return p[f * 32]; }
};
struct FisherShared {
  fx tape[kTapeSlots][kFtAll][32];
  fx col[kFxSums][kFisherFxThreads];           // the forward's sums (unused), then the seeds, a column per thread
  double J[kFisherWarps][PE_NPARAM][32];       // rows Re/Im of A', E', T'
  double gJ[kFisherWarps][PE_NPARAM][32];      // the same times the channel's 4 / (T S)
  alignas(16) fx pc[kFxProjAll];
  double rot[3][3];                            // d(lambda, beta, psi) per rotation cotangent
  long long next;
};
__global__ void __launch_bounds__(kFisherFxThreads, 2) k_fisher_fx(DetSet ds, int B, const SampleCoef* __restrict__ coef,
                                                                   const SampleGrad* __restrict__ sgrad,
                                                                   const int* __restrict__ nend,
                                                                   const long long* __restrict__ off, double* part, int split,
                                                                   unsigned long long* ctr) {
  extern __shared__ __align__(16) unsigned char fisher_smem[];
  FisherShared& sm = *reinterpret_cast<FisherShared*>(fisher_smem);
  const int P = ds.ndet * B;
  const long long total = off[P] * split;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  fx* col = &sm.col[0][threadIdx.x];
  for (long long t = blockIdx.x, tn = 0; t < total; t = work_next(tn, &sm.next)) {
    tn = work_fetch(ctr, t);
    const long long tile = t / split;
    const int p = find_pair_warp(off, P, tile);
    if (!PE_CHK(p >= 0 && p < P && off[p + 1] * split <= total && nend[p] <= ds.d[p / B].nb, 64)) continue;
    const int I = p / B, s = p - I * B;
    const DetDev& D = ds.d[I];
    const SampleCoef& S = coef[s];
    const SampleGrad& SG = sgrad[s];
    fx_proj_prologue(D, S, sm.pc);
    if (threadIdx.x >= 64 && threadIdx.x < 73) {
      const int j = (threadIdx.x - 64) / 3, c = (threadIdx.x - 64) % 3;
      const double W[3] = {c == 0 ? 1.0 : 0.0, c == 1 ? 1.0 : 0.0, c == 2 ? 1.0 : 0.0};
      double a = 0.0;
      for (int i = 0; i < 3; ++i)
        a += rotation_to_frame(S, W, 0, i) * SG.dk[i][j] + rotation_to_frame(S, W, 1, i) * SG.dp[i][j];
      sm.rot[j][c] = a;
    }
    fx_proj3(sm.pc);
    double own = 0.0;   // this lane's entry (fisher_lane_entry), summed over the passes
    const int subs = kTileBins / 32 / split, sub0 = int(t - tile * split) * subs;
#pragma unroll 1
    for (int sub = sub0; sub < sub0 + subs; ++sub) {
      const int b = int(tile - off[p]) * kTileBins + sub * 32 + lane;
      const bool on = b < nend[p];
      FxBin Bn;
      double fm13 = 0.0;
      if (on) {
        load_bin_fx(D, b, S.tc, Bn);
        fm13 = D.fm13[b];
#pragma unroll 1
        for (int md = 0; md < kNModes; ++md) {
          const ModeCoef& C = S.md[md];
          if (tape_slot(md) != w || (md == 3 && S.pair32) || !C.active || !dlt_pos(Bn.f, C.fend)) continue;
          const ModeCoef* C2 = (md == 0 && S.pair32) ? &S.md[3] : nullptr;
          const FisherTape tp = {&sm.tape[w][0][lane]};
          FxAccT<kFisherFxThreads> a;
          fx_zero(a, col);
          mode_bin_fx(D, S, C, Bn, a, ds.d[0].fcis, ds.d[0].fsinc, sm.pc, md, C2, tp);
          const double v = C.cm * Bn.f13, tw = __longlong_as_double(tp.ld(kFtW)), amp = __longlong_as_double(tp.ld(kFtAmp0)) * tw;
          double2 Ap, Ac;
          fx_weights(S, C, C2, amp, v, Ap, Ac);
          const FxChain h = fx_chain(D, S, SG, C, SG.md[md], Bn, fm13, v, tw, tp.ld(kFtC), tp.ld(kFtS));
          const double f[12] = {h.dv, h.ddv, h.pq, h.dq, h.iv, h.co, h.so, h.tap, Ap.x, Ap.y, Ac.x, Ac.y};
#pragma unroll
          for (int i = 0; i < 12; ++i) tp.st(kFtChain + i, __double_as_longlong(f[i]));
        }
      }
      __syncthreads();   // the tape is written; the last pass's readers of J and gJ are done
      double row[PE_NPARAM];
#pragma unroll
      for (int i = 0; i < PE_NPARAM; ++i) row[i] = 0.0;
      if (on) {
        double2 bb[3], pq[6];
        for (int c = 0; c < 3; ++c) bb[c] = make_double2(w == 2 * c ? 1.0 : 0.0, w == 2 * c + 1 ? 1.0 : 0.0);
        const double2 sc = D.sca[b];
        link_seeds<1>(bb, sc.x, sc.y, pq);
        const int Es = fx_seeds<kFisherFxThreads>(pq, col);
        const fx a3 = fx_times_k((unsigned)(D.k0 + b), D.fx_a3);
        const double invf = fm13 * fm13 * fm13, n2pif = -2.0 * kPi * Bn.f, fR = -D.R * n2pif;
        FxBinAcc ga;
        ga.zero();
#pragma unroll 1
        for (int md = 0; md < kNModes; ++md) {
          if ((md == 3 && S.pair32) || Es == 0 || !S.md[md].active || !dlt_pos(Bn.f, S.md[md].fend)) continue;
          const FisherTape tp = {&sm.tape[tape_slot(md)][0][lane]};
          mode_bwd_fx<kFisherFxThreads>(D, S, SG, md, (md == 0 && S.pair32) ? 3 : -1, Bn, fm13, invf, fR, n2pif, a3, col, Es, ga, sm.pc, tp);
        }
        GradAcc g;
        fx_bin_grad(S, SG, ga, g);
        row[0] = g.M; row[1] = g.q; row[2] = g.c1; row[3] = g.c2; row[4] = g.dL; row[5] = g.io; row[6] = g.ph; row[10] = g.tc;
#pragma unroll
        for (int j = 0; j < 3; ++j) row[7 + j] = fma(sm.rot[j][0], g.k[0], fma(sm.rot[j][1], g.k[1], sm.rot[j][2] * g.k[2]));
      }
      const double gg = on ? D.gg[(w >> 1) * D.nb + b] : 0.0;
#pragma unroll
      for (int i = 0; i < PE_NPARAM; ++i) {
        sm.J[w][i][lane] = row[i];
        sm.gJ[w][i][lane] = gg * row[i];
      }
      __syncthreads();
      // entries e = w, w + 6, ... of the upper triangle, row by row
      double F[kFisherW / kFisherWarps];
#pragma unroll
      for (int e = 0; e < kFisherW / kFisherWarps; ++e) F[e] = 0.0;
#pragma unroll 1
      for (int r = 0; r < kFisherWarps; ++r) {
        int i = 0, k = w;
        while (k >= PE_NPARAM - i) { k -= PE_NPARAM - i; ++i; }
#pragma unroll
        for (int e = 0; e < kFisherW / kFisherWarps; ++e) {
          F[e] = fma(sm.gJ[r][i][lane], sm.J[r][i + k][lane], F[e]);
          k += kFisherWarps;
          while (i < PE_NPARAM && k >= PE_NPARAM - i) { k -= PE_NPARAM - i; ++i; }
        }
      }
      own += fisher_lane_sum(F, lane);
    }
    const int e = fisher_lane_entry(lane);
    if (e >= 0) part[t * kFisherW + w + kFisherWarps * e] = own;
  }
  work_done(ctr);
}

// Per point: thread (r, e) adds entry e of the tiles r, r + 8, ... over the detectors, then thread e its eight rows. A tile's sum is that of its
// items (split of them) in order, as k_fisher_fx adds the passes of an undivided tile, so the bits do not depend on the split.
constexpr int kFisherRows = 8;
__global__ void __launch_bounds__(kFisherW * kFisherRows) k_fisher_reduce(DetSet ds, int B, const long long* off, const double* part,
                                                                        const SampleCoef* coef, int split, double* F) {
  __shared__ double red[kFisherRows][kFisherW];
  const int s = blockIdx.x;
  const int e = threadIdx.x % kFisherW, r = threadIdx.x / kFisherW;
  double a = 0.0;
  for (int I = 0; I < ds.ndet; ++I) {
    const int p = I * B + s;
    if (!PE_CHK(off[p] >= 0 && off[p + 1] <= off[ds.ndet * B], 128)) continue;
    for (long long t = off[p] + r; t < off[p + 1]; t += kFisherRows) {
      double x = part[t * split * kFisherW + e];
      for (int k = 1; k < split; ++k) x += part[(t * split + k) * kFisherW + e];
      a += x;
    }
  }
  red[r][e] = a;
  __syncthreads();
  if (r != 0) return;
  for (int k = 1; k < kFisherRows; ++k) a += red[k][e];
  if (!coef[s].valid) a = 0.0;
  int i = 0, k = 0, idx = e;
  while (idx >= PE_NPARAM - i) { idx -= PE_NPARAM - i; ++i; }
  k = i + idx;
  F[(size_t)s * 121 + i * PE_NPARAM + k] = a;
  F[(size_t)s * 121 + k * PE_NPARAM + i] = a;
}

cudaError_t launch_prep_grad(const double* theta, int B, unsigned mask, const DetSet& ds, SampleCoef* coef,
                             SampleGrad* sgrad, int* nend, int* status, cudaStream_t st) {
  return prep_launch<true>(theta, B, mask, ds, coef, sgrad, nend, status, st);
}
cudaError_t launch_grad_fwd(const DetSet& ds, int B, const SampleCoef* coef, const SampleGrad* sgrad, const int* nend,
                            const long long* off, double* part, int grid, bool mixed, double* tape, unsigned long long* ctr,
                            cudaStream_t st) {
  if (fx_all_ok(ds))
    k_grad_fwd_fx<<<grid, kTileBins, 0, st>>>(ds, B, coef, sgrad, nend, off, part, tape, ctr);
  else if (mixed)
    k_grad_fwd_mixed<<<grid, kTileBins, 0, st>>>(ds, B, coef, sgrad, nend, off, part, tape);
  else
    k_grad_fwd_tape<<<grid, kTileBins, 0, st>>>(ds, B, coef, sgrad, nend, off, part, tape);
  return pe::launch_status();
}
cudaError_t launch_grad_reduce(const DetSet& ds, int B, const long long* off, const double* part,
                               const SampleCoef* coef, const SampleGrad* sgrad, double* logl, double* grad,
                               cudaStream_t st) {
  bool small = true;
  for (int i = 0; i < ds.ndet; ++i) small &= (ds.d[i].nb + kTileBins - 1) / kTileBins <= kGradWarpTiles;
  if (small)
    k_grad_reduce_warp<<<(unsigned)(((long long)B * 32 + 127) / 128), 128, 0, st>>>(ds, B, off, part, coef, sgrad, logl, grad);
  else
    k_grad_reduce<<<B, kGradW * 32, 0, st>>>(ds, B, off, part, coef, sgrad, logl, grad);
  return pe::launch_status();
}
// Items per 128-bin tile: a few points leave the chip's SMs two or three tiles each, so up to 32 possible tiles per SM the fixed-point
// kernel's items are a quarter tile; beyond, whole tiles (a quarter of the partials). Whole and quarter tiles, whole calls with every bin
// active: 8 tiles 265 and 113 us, 128 267 and 203, 1,024 1072 and 1020, 2,048 2015 and 1971, 4,096 3783 and 3871, 8,192 7481 and 7672. Samples over
// the prior leave most of a long grid's tiles without work, and quarters win for longer.
int fisher_split(const DetSet& ds, long long max_tiles, int sms) { return fx_all_ok(ds) && max_tiles <= 32LL * sms ? 4 : 1; }
cudaError_t launch_fisher_fwd(const DetSet& ds, int B, const SampleCoef* coef, const SampleGrad* sgrad,
                              const int* nend, const long long* off, double* part, long long max_tiles, int sms, int split,
                              unsigned long long* ctr, cudaStream_t st) {
  if (fx_all_ok(ds)) {
    cudaError_t e = cudaFuncSetAttribute(k_fisher_fx, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(FisherShared));
    if (e != cudaSuccess) return e;
    const int grid = (int)std::max(1LL, std::min(max_tiles * split, 2LL * sms));
    k_fisher_fx<<<grid, kFisherFxThreads, sizeof(FisherShared), st>>>(ds, B, coef, sgrad, nend, off, part, split, ctr);
  } else {
    const int grid = (int)std::max(1LL, std::min(max_tiles, 16LL * sms));
    k_fisher_fwd<<<grid, 32 * kFisherWarps, 0, st>>>(ds, B, coef, sgrad, nend, off, part);
  }
  return pe::launch_status();
}
cudaError_t launch_fisher_reduce(const DetSet& ds, int B, const long long* off, const double* part,
                                 const SampleCoef* coef, int split, double* F, cudaStream_t st) {
  k_fisher_reduce<<<B, kFisherW * kFisherRows, 0, st>>>(ds, B, off, part, coef, split, F);
  return pe::launch_status();
}
int grad_partial_width() { return kGradW; }
// FP64: two CTAs per SM (230 registers, no spills; three, at 168 registers, ran 0.4 % slower);
// mixed: three (168 registers, a few hundred bytes of spills), which its latency-bound sweep
// prefers (33.6k against 30.9k grad evals/s with two, 33.0k with four)
// Fixed point: kGradFxCtas.
int grad_tape_ctas_per_sm(const DetSet& ds, bool mixed) { return fx_all_ok(ds) ? kGradFxCtas : (mixed ? 3 : 2); }
size_t grad_tape_doubles_per_cta() { return (size_t)kTapeDoubles; }
int fisher_partial_width() { return kFisherW; }

// Index-check error word of this file's kernels (checked build; 0 otherwise), cleared when read.
int checked_take_grad() { return pe_checked_take_local(); }

}  // namespace pe

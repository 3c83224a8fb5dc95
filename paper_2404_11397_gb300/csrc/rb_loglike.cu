// rb_loglike.cu -- batched relative-binning log-likelihood and its adjoint
// (steps a3-a6): ratio at the bin edges, per-bin linearisation, contraction
// with the summary data, and the reverse sweep back to the 13 parameters.
//
// Relative binning (Sec. II.C, Eqs. 4-5): per detector d,
//   r(f_e) = rho_d exp(-2 pi i x_d(f_e)),   x_d = dPsi_d / (2 pi)  [turns]
//   r0(b) = (r_b + r_{b+1}) / 2,  r1(b) = (r_{b+1} - r_b) / (f_{b+1} - f_b)
//   <d|h> = Re sum_b [A0 r0* + A1 r1*],  <h|h> = sum_b [B0 |r0|^2 + 2 B1 Re(r0 r1*)].
// The kernels evaluate the deviation from the fiducial point: with
// r = 1 + delta, s = delta_b + delta_{b+1}, t = delta_{b+1} - delta_b,
//   log L = base + sum_{d,b} Re(alpha0 s*) + Re(alpha1 t*) - beta0 (Re s + |s|^2/4)
//                            - beta1 (Re t + Re(s t*)/2),
// alpha0 = A0/2, alpha1 = A1/df_b, beta0 = B0/2, beta1 = B1/df_b and the FP64
// constant base = sum_d (Re sum_b A0 - sum_b B0/2) = log L(theta_ref).  At the
// fiducial point delta = 0 exactly and the result is base, bit for bit.
// With the Newtonian amplitude the ratio has the same modulus |rho_d| at every
// edge, so Re(r0 r1*) = (|r_{b+1}|^2 - |r_b|^2) / (2 df_b) = 0: the beta1 term
// (Re t + Re(s t*)/2 = (|1 + delta_{b+1}|^2 - |1 + delta_b|^2) / 2) and its
// derivatives vanish identically.  The kernels leave it out (in FP32 it is
// rounding noise about zero; in FP64 leaving it out changes results by 1e-14).
// delta is formed without cancellation from the half angle:
//   exp(-2 pi i x) - 1 = -2 sin^2(pi x) - 2 i sin(pi x) cos(pi x),
//   delta = rho (exp(-2 pi i x) - 1) + (rho - 1).
//
// Mapping: one warp per walker (persistent: each block takes a contiguous,
// equal share of the walkers and its warps take them in turn).  Float-float
// path: in iteration i lane l holds edges 63 i + 2 l and 63 i + 2 l + 1 and
// the bins on their right as the two halves of paired FP32 values (the slot
// image, EventDev::slot32); FP64-phase path: lane l handles edge 31 c + l of
// chunk c and bin 31 c + l (lanes 0..30).  Either way a bin's right edge is
// at most one shuffle away and consecutive iterations overlap by one edge.
// Edge and bin tables live in shared memory.  The adjoint reuses the same
// mapping: each edge collects the cotangent from its own bin and from the
// bin on its left; an edge shared by two iterations collects the two halves
// in two passes, which is exact because the adjoint is linear in the per-edge
// cotangent.
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "rb_internal.cuh"
#include "rb_setup_dd.cuh"

namespace rb {

#ifndef RB_MIXED_THREADS
#define RB_MIXED_THREADS 512
#endif
constexpr int kThreads = RB_MIXED_THREADS;  // threads per block of the mixed likelihood kernel
constexpr unsigned kFull = 0xffffffffu;
// The current walker's constants sit in shared memory (read by broadcast
// loads in every iteration instead of held in registers): as the set-up wrote
// them (WalkerMixed: float4 quads, detectors 0 and 1 paired, detector D - 1
// alone when D is odd), and for the float-float loop expanded into {x, x, y, y}
// quads (WarpSlot::dup).

// Shared-memory load that the compiler may not hoist out of a loop.
__device__ __forceinline__ float4 lds4(const float4* p) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"((unsigned)__cvta_generic_to_shared(p)));
  return v;
}

// Asynchronous global -> shared copies (cp.async): the copies of a thread
// complete, in issue order, by its next cp_async_wait_all().
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem)
               : "memory");
}
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Per-warp shared-memory slot after the tables: two buffers for a walker's
// set-up record (its constants, WalkerMixed) and tangents, so that the next
// walker's are fetched while this one runs.
constexpr int kTanBytes = 384;
// what a warp needs besides its walker's record and tangents
struct __align__(16) WarpWork {
  float red[32];  // the walker's adjoint sums
  // the current walker's constants, each value in both halves of a pair
  // (float-float path): {hi, hi, lo, lo} of dc_k (k < kNBasis), then per
  // detector {tau_hi, tau_hi, tau_lo, tau_lo}, {rho_r, rho_r, rho_i, rho_i},
  // {sig_r, sig_r, sig_i, sig_i}, and last the walker's rounding constant m
  // of the phase sums (split_acc) in all four
  float4 dup[kNBasis + 3 * kMaxDet + 1];
  // per lane: the bound on |g_k| or f that the lane's phase term takes in the
  // record expansion (constant over the launch)
  float lane_gmax[32];
};
struct __align__(16) WarpSlot {
  WalkerMixed rec[2];
  unsigned char tan[2][kTanBytes];
  WarpWork work;
};
// Shared memory of a FUSED block after the tables: its walkers' records and
// tangents, then the set-up's values, whose space the warps take over.
struct __align__(16) FusedRecords {
  WalkerMixed rec[kSetupWalkers];
  WalkerTan<float> tan[kSetupWalkers];
  unsigned long long tan_done;  // mbarrier: the tangent warps, once each
};

// One-shot mbarrier in shared memory: count arrivals complete its phase 0.
__device__ __forceinline__ void mbar_init(unsigned long long* b, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* b) {
  asm volatile("{.reg .b64 t;\n\tmbarrier.arrive.shared::cta.b64 t, [%0];}" ::"r"((unsigned)__cvta_generic_to_shared(b)) : "memory");
}
// Waits for phase 0, at most kMbarTries attempts (a fraction of a second; the
// arrivals are unconditional, so the limit is not met): false if it gave up.
constexpr int kMbarTries = 1 << 16;
__device__ __forceinline__ bool mbar_wait(unsigned long long* b) {
  for (int i = 0; i < kMbarTries; ++i) {
    unsigned ok;
    asm volatile("{.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\tselp.u32 %0, 1, 0, p;}"
                 : "=r"(ok)
                 : "r"((unsigned)__cvta_generic_to_shared(b))
                 : "memory");
    if (ok) return true;
  }
  return false;
}
constexpr size_t kFusedWork = sizeof(DdSmem) > (kThreads / 32) * sizeof(WarpWork) ? (sizeof(DdSmem) + 15) / 16 * 16
                                                                               : (kThreads / 32) * sizeof(WarpWork);
constexpr size_t kFusedBytes = sizeof(FusedRecords) + kFusedWork;
static_assert(kFusedBytes % 16 == 0, "the MALA chains start on a 16-byte boundary");
static_assert(sizeof(FusedRecords) % 16 == 0, "the set-up's values start on a 16-byte boundary");
static_assert(kThreads > kDdRoleThreads && kThreads >= kTanWarps * 32, "a FUSED block has a warp for every set-up role");
static_assert(sizeof(WalkerMixed) % 16 == 0, "record copied in 16-byte pieces");
static_assert(sizeof(WalkerTan<float>) <= kTanBytes && sizeof(WalkerTan<float>) % 8 == 0, "tangent buffer");

// Issue (the whole warp) the copies of one walker's record (unless PHASE64,
// whose FP64 record is read directly) and tangents into buffer buf, as one
// cp.async group.  Global addresses: records 16-byte, tangents 8-byte
// aligned (checked by the launcher).
template <bool GRAD, bool PHASE64>
__device__ __forceinline__ void prefetch_walker(WarpSlot* slot, int buf, const void* rec, const void* tan, int lane) {
  if (!PHASE64 && lane < (int)(sizeof(WalkerMixed) / 16))
    cp_async16(reinterpret_cast<unsigned char*>(&slot->rec[buf]) + 16 * lane, static_cast<const unsigned char*>(rec) + 16 * lane);
  if (GRAD) {
    constexpr int n = (int)(sizeof(WalkerTan<float>) / 8);
#pragma unroll
    for (int i = lane; i < n; i += 32) cp_async8(slot->tan[buf] + 8 * i, static_cast<const unsigned char*>(tan) + 8 * i);
  }
  cp_async_commit();
}

// Exact float -> double conversion on the integer pipe: an SMSP's FP64 unit
// takes ~65 clocks per warp instruction, conversions included, and the warps
// of a block reach their epilogues together.  Normal numbers: the exponent
// rebiased by 1023 - 127 and the mantissa moved up 29 bits; zero, subnormals,
// infinities and NaN take the regular conversion.
__device__ __forceinline__ double f2d_int(float x) {
  const unsigned u = __float_as_uint(x), m = u & 0x7fffffffu;
  if (m - 0x00800000u < 0x7f000000u)
    return __hiloint2double((int)((u & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(m << 29));
  return (double)x;
}

// Float-pair warp sum: (h, l) on entry is a lane's value as an unevaluated
// sum; every lane returns the warp total (two-sum of the high parts, the low
// parts added, renormalised at each step), all on the FP32 pipe.
__device__ __forceinline__ void warp_sum_ff(float& h, float& l) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float oh = __shfl_xor_sync(0xffffffffu, h, o), ol = __shfl_xor_sync(0xffffffffu, l, o);
    const float s = __fadd_rn(h, oh);
    const float bb = __fsub_rn(s, h);
    const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(s, bb)), __fsub_rn(oh, bb));
    const float lo = __fadd_rn(__fadd_rn(l, ol), e);
    h = __fadd_rn(s, lo);
    l = __fsub_rn(lo, __fsub_rn(h, s));
  }
}

// Adds the float pair (bh, bl) to (h, l) (two-sum of the high parts).
__device__ __forceinline__ void ff_add(float& h, float& l, float bh, float bl) {
  const float s = __fadd_rn(h, bh);
  const float bb = __fsub_rn(s, h);
  const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(s, bb)), __fsub_rn(bh, bb));
  const float lo = __fadd_rn(__fadd_rn(l, bl), e);
  h = __fadd_rn(s, lo);
  l = __fsub_rn(lo, __fsub_rn(h, s));
}

struct LaunchArgs {
  EventDev ev;
  const void* ws;    // WalkerMixed* or WalkerF64*
  const void* tan;   // WalkerTan<float>* or WalkerTan<double>*
  int64_t W;
  double* logl;
  double* grad;
  MalaArgs mala;     // MALA kernels only
};
// the FUSED kernels form the records themselves (a MALA step's from its proposals, theta NULL)
struct FusedArgs : LaunchArgs {
  const double* theta;  // [W][13]
  EventConst ec;
};

// MALA accept/reject for walker w after its log L and d log L / d theta
// (lane j < 13 holds component j): gradient in sampling coordinates,
//   log alpha = log pi(z') - log pi(z) - 1/2 sum_j [(xi_j + eps_j (g_j + g'_j)/2)^2 - xi_j^2]
// (Sec. II.D, MALA; the sum over j is a warp reduction), accept when
// log u < log alpha, and the chain state updated in place.  The whole warp
// calls it (logl and inside are warp-uniform).
struct MalaWalker {
  bool inside;
  double lu, jac9, jac12;  // log u, the Jacobian factors of cos iota and sin dec
  double zp;               // the lane's component of the proposal
};
__device__ __forceinline__ MalaWalker mala_walker(const MalaArgs& m, int64_t w, int lane) {
  return {m.inside[w] != 0, m.lu[w], m.jac[2 * w], m.jac[2 * w + 1], lane < kNPar ? m.zp[w * kNPar + lane] : 0.0};
}
__device__ __forceinline__ void mala_finish(const MalaArgs& m, int64_t w, int lane, double logl, double gth,
                                            const MalaWalker& mw) {
  const bool inside = mw.inside;
  const double logpp = inside ? logl : -INFINITY;
  double gz = 0.0, term = 0.0;
  if (lane < kNPar) {
    gz = gth;
    if (lane == 9) gz = gth * mw.jac9;
    else if (lane == 12) gz = gth * mw.jac12;
    if (!inside) gz = 0.0;
  }
  if (m.init) {
    if (lane < kNPar) m.gz[w * kNPar + lane] = gz;
    if (lane == 0) {
      m.logp[w] = logpp;
      if (m.accepted) m.accepted[w] = inside ? 1 : 0;
    }
    return;
  }
  if (lane < kNPar) {
    const double xi = m.xi[w * kNPar + lane];
    const double t = xi + 0.5 * m.eps[lane] * (m.gz[w * kNPar + lane] + gz);
    term = t * t - xi * xi;
  }
  term = warp_sum_f64(term);
  const double la = (logpp == -INFINITY) ? -INFINITY : logpp - m.logp[w] - 0.5 * term;
  const bool acc = mw.lu < la;
  if (acc) {
    if (lane < kNPar) {
      m.z[w * kNPar + lane] = mw.zp;
      m.gz[w * kNPar + lane] = gz;
    }
    if (lane == 0) m.logp[w] = logpp;
  }
  if (lane == 0 && m.accepted) m.accepted[w] = acc ? 1 : 0;
}

// The proposals of a FUSED block's chains, in its shared memory (as
// k_mala_propose forms them, expression for expression).
struct __align__(16) MalaBlock {
  double theta[kSetupWalkers][kNPar];  // theta(z'), or theta(z) outside the box
  double zp9[kSetupWalkers], zp12[kSetupWalkers];  // cos iota and sin dec of the proposal (its other components are theta's)
  double lu[kSetupWalkers], jac9[kSetupWalkers], jac12[kSetupWalkers];
  int inside[kSetupWalkers];
};
// The whole block calls it; n chains from w0.  The block is synchronised at its end.
__device__ __forceinline__ void mala_propose_block(const MalaArgs& m, int64_t w0, int n, MalaBlock& S) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < kSetupWalkers) S.inside[tid] = 1;
  __syncthreads();
  for (int i = tid; i < n * kNPar; i += kThreads) {
    const int l = i / kNPar, j = i - l * kNPar;
    const int64_t g = w0 * kNPar + i;
    const double c = m.z[g];
    const double p = m.init ? c : c + 0.5 * m.eps[j] * m.eps[j] * m.gz[g] + m.eps[j] * m.xi[g];
    S.theta[l][j] = p;
    if (j == 9) S.zp9[l] = p;
    if (j == 12) S.zp12[l] = p;
    if (!(p > m.lo[j] && p < m.hi[j])) S.inside[l] = 0;
  }
  __syncthreads();
  // a chain outside the box is evaluated at its current state (and rejected)
  for (int i = tid; i < n * kNPar; i += kThreads) {
    const int l = i / kNPar, j = i - l * kNPar;
    if (S.inside[l] == 0 && j != 9 && j != 12) S.theta[l][j] = m.z[w0 * kNPar + i];
  }
  // the FP64 functions of a chain on four warps side by side, one per SM sub-partition
  if (warp < 4 && lane < n) {
    const bool in = S.inside[lane] != 0;
    const double* zw = m.z + (w0 + lane) * kNPar;
    const double p9 = S.zp9[lane], p12 = S.zp12[lane];
    if (warp == 0) {
      S.theta[lane][9] = acos(in ? p9 : zw[9]);
    } else if (warp == 1) {
      S.theta[lane][12] = asin(in ? p12 : zw[12]);
    } else if (warp == 2) {
      // d iota / d cos iota = -1 / sin iota, d dec / d sin dec = 1 / cos dec
      // (1 - z^2 as (1 - z)(1 + z): no cancellation next to the box edges)
      S.jac9[lane] = in ? -1.0 / sqrt((1.0 - p9) * (1.0 + p9)) : 0.0;
      S.jac12[lane] = in ? 1.0 / sqrt((1.0 - p12) * (1.0 + p12)) : 0.0;
    } else {
      S.lu[lane] = m.init ? 0.0 : log(m.u[w0 + lane]);
    }
  }
  __syncthreads();
}

// Chain rule for one walker: lane j < 13 returns d log L / d theta_j from the
// reduced adjoints (adj_c over the basis coefficients, adj_tau per detector
// delay, G_d = conj(gbar_rho_d) rho_d per prefactor: d log L = Re(G_d dln rho_d))
// and the set-up tangents.  Every lane runs one instruction stream (the lane's
// tangent entries picked by index and select, no divergent branches).
__device__ __forceinline__ float madd(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double madd(double a, double b, double c) { return fma(a, b, c); }
template <int D, class T>
__device__ __forceinline__ T chain_rule_lanes(int j, const T* adj_c, const T* adj_tau, const T (*G)[2],
                                              const WalkerTan<T>& tn) {
  const T* t = reinterpret_cast<const T*>(&tn);
  constexpr int oDc = offsetof(WalkerTan<T>, dc) / sizeof(T), oPhi = offsetof(WalkerTan<T>, dphi0) / sizeof(T);
  constexpr int oDtd = offsetof(WalkerTan<T>, dtd) / sizeof(T), oLnP = offsetof(WalkerTan<T>, dlnP) / sizeof(T);
  constexpr int oMc = offsetof(WalkerTan<T>, lnamp_Mc) / sizeof(T), oDl = offsetof(WalkerTan<T>, lnamp_dL) / sizeof(T);
  const bool intr = j < kNTanIntr, radec = j == 11 || j == 12, ext = j >= 9;
  const int ji = intr ? j : 0, jr = radec ? j - 11 : 0, je = ext ? j - 9 : 0;
  T g = T(0);
#pragma unroll
  for (int k = 0; k < kNBasis; ++k) {
    const T v = t[oDc + k * kNTanIntr + ji];
    g = madd(adj_c[k], intr ? v : T(0), g);
  }
  // d ln rho_d = lr + i li: ln amplitude (Mc, dL), -dPhi0 (Mc, q), phi_c, antenna (iota, psi, ra, dec)
  const int ir = j == 0 ? oMc : (j == 6 ? oDl : oMc);
  const T lr_own = (j == 0 || j == 6) ? t[ir] : T(0);
  const int ii = j == 1 ? oPhi + 1 : oPhi;
  const T li_own = (j == 0 || j == 1) ? -t[ii] : (j == 8 ? T(1) : T(0));
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const T td = t[oDtd + 2 * d + jr];
    g = madd(adj_tau[d], radec ? td : (j == 7 ? T(1) : T(0)), g);
    const T pr = t[oLnP + 8 * d + 2 * je], pi = t[oLnP + 8 * d + 2 * je + 1];
    const T lr = ext ? pr : lr_own, li = ext ? pi : li_own;
    g += G[d][0] * lr - G[d][1] * li;  // Re(G_d dln rho_d)
  }
  return g;
}

namespace pv {
// Per-walker detector constants and adjoint accumulators of one detector
// (V = float) or of the detector pair 0, 1 (V = float2).
template <class V>
struct DetState {
  V tau_h, tau_l;          // delta tau [s] as a float pair
  V rho_r, rho_i, sig_r, sig_i;
  V acc, acc_lo;           // log L terms, float-pair accumulator
  V adj_tau, adj_rr, adj_ri;
};

// One bin edge (and the bin on its right) for one detector or a detector
// pair: half-angle sin/cos, delta = rho (e^{-2 pi i y} - 1) + sigma, the
// neighbour edge by a shuffle, the bin's contraction with the tables (bins
// of lanes 0..30) and, with GRAD, the edge cotangent.  Returns d log L / dy
// per detector (times 1/2pi) for the basis adjoint.  The whole warp calls it.
template <bool GRAD, class V>
__device__ __forceinline__ V det_edge(V y, DetState<V>& st, const V* bt, bool has_bin, bool has_edge, int lane, V fe) {
  V sn, cs;
  sincos_half(y, sn, cs);
  const V t2 = mul(splat<V>(-2.f), sn);
  const V em_r = mul(t2, sn), em_i = mul(t2, cs);  // e^{-2 pi i y} - 1
  const V dr = fma(st.rho_r, em_r, fma(neg(st.rho_i), em_i, st.sig_r));
  const V di = fma(st.rho_r, em_i, fma(st.rho_i, em_r, st.sig_i));
  const V nr = shfl_down(dr), ni = shfl_down(di);
  V Ur = splat<V>(0.f), Ui = Ur, Vr = Ur, Vi = Ur;
  if (has_bin) {
    // bt: alpha0 (re, im), alpha1 (re, im), -beta0 (the -beta1 entry is not
    // needed: the beta1 term vanishes for a ratio of constant modulus)
    const V sr = add(dr, nr), si = add(di, ni), tr = sub(nr, dr), ti = sub(ni, di);
    V v = mul(bt[0], sr);
    v = fma(bt[1], si, v);
    v = fma(bt[2], tr, v);
    v = fma(bt[3], ti, v);
    v = fma(bt[4], fma(splat<V>(0.25f), fma(sr, sr, mul(si, si)), sr), v);
    const V s = add(st.acc, v);  // two-sum into (acc, acc_lo)
    const V bb = sub(s, st.acc);
    st.acc_lo = add(st.acc_lo, add(sub(st.acc, sub(s, bb)), sub(v, bb)));
    st.acc = s;
    if (GRAD) {
      const V hs_r = fma(splat<V>(0.5f), sr, splat<V>(1.f)), hs_i = mul(splat<V>(0.5f), si);  // 1 + s/2
      Ur = fma(bt[4], hs_r, bt[0]);
      Ui = fma(bt[4], hs_i, bt[1]);
      Vr = bt[2];
      Vi = bt[3];
    }
  }
  V dldx = splat<V>(0.f);
  if (GRAD) {
    V gr = sub(Ur, Vr), gi = sub(Ui, Vi);  // own bin (edge on its left)
    const V lr = shfl_up(add(Ur, Vr)), li = shfl_up(add(Ui, Vi));
    if (lane > 0) {
      gr = add(gr, lr);
      gi = add(gi, li);
    }
    if (has_edge) {
      const V rr = add(splat<V>(1.f), dr);
      dldx = fma(gr, di, mul(neg(gi), rr));  // Im(conj(gbar) r); times 2 pi later
      st.adj_tau = fma(dldx, fe, st.adj_tau);
      const V Er = add(splat<V>(1.f), em_r);  // gbar_rho += gbar conj(E)
      st.adj_rr = fma(gr, Er, fma(gi, em_i, st.adj_rr));
      st.adj_ri = fma(gi, Er, fma(neg(gr), em_i, st.adj_ri));
    }
  }
  return dldx;
}
// The same for the two edges of a slot (halves A and B: edges e_A = 63 i + 2 l
// and e_B = e_A + 1 of lane l) and one detector: e_A's right neighbour is
// the lane's own e_B, e_B's is lane l + 1's e_A (one shuffle); e_B's left
// bin is the lane's own A bin, e_A's is lane l - 1's B bin, none for lane 0
// (its e_A is lane 31's e_B of the previous iteration, which collected it).
// Edges without a bin, and slots past the last edge, have zero tables, so
// they add nothing.  vsum collects the bin terms of log L, adj_x
// d log L / dy (times 1/2pi) for the basis adjoint, (adj_rr, adj_ri) the sum
// of conj(gbar) r over the edges (the prefactor's adjoint times rho: G_d).
// The bin's term in the coefficients of its edge values (q0 = {gmr, gpr},
// q1 = {gmi, gpi}, q2 = {h, q} of the slot image): with d = delta at the
// left edge and n at the right one,
//   Re(alpha0 s*) + Re(alpha1 t*) - beta0 (Re s + |s|^2/4)
//     = gmr dr + gpr nr + gmi di + gpi ni + q |s|^2,
// and the cotangents of the left and right edge values are
//   (gmr + h sr, gmi + h si) and (gpr + h sr, gpi + h si).
template <bool GRAD>
__device__ __forceinline__ void det_edge_slot(float2 y, float4 rho, float4 sig, const float2 (&bt)[6], int lane,
                                              float2 fe, float2& vsum, float2& adj_x, float& adj_tau, float& adj_rr,
                                              float& adj_ri) {
  const float2 rho_r = make_float2(rho.x, rho.y), rho_i = make_float2(rho.z, rho.w);
  const float2 sig_r = make_float2(sig.x, sig.y), sig_i = make_float2(sig.z, sig.w);
  float2 sn, cs;
  sincos_half(y, sn, cs);
  const float2 t2 = mul(splat<float2>(-2.f), sn);
  const float2 em_r = mul(t2, sn), em_i = mul(t2, cs);  // e^{-2 pi i y} - 1
  const float2 dr = fma(rho_r, em_r, fma(neg(rho_i), em_i, sig_r));
  const float2 di = fma(rho_r, em_i, fma(rho_i, em_r, sig_i));
  const float2 nr = make_float2(dr.y, __shfl_down_sync(0xffffffffu, dr.x, 1));
  const float2 ni = make_float2(di.y, __shfl_down_sync(0xffffffffu, di.x, 1));
  // bt: gmr, gpr, gmi, gpi, h, q (the beta1 term vanishes for a ratio of
  // constant modulus)
  const float2 sr = add(dr, nr), si = add(di, ni);
  float2 v = mul(bt[0], dr);
  v = fma(bt[1], nr, v);
  v = fma(bt[2], di, v);
  v = fma(bt[3], ni, v);
  v = fma(bt[5], fma(sr, sr, mul(si, si)), v);
  vsum = add(vsum, v);
  if (GRAD) {
    float2 gr = fma(bt[4], sr, bt[0]), gi = fma(bt[4], si, bt[2]);  // own bin (edge on its left)
    const float2 pr = fma(bt[4], sr, bt[1]), pi = fma(bt[4], si, bt[3]);  // the bin's right edge
    const float lr = __shfl_up_sync(0xffffffffu, pr.y, 1), li = __shfl_up_sync(0xffffffffu, pi.y, 1);
    gr = add(gr, make_float2(lane == 0 ? 0.f : lr, pr.x));
    gi = add(gi, make_float2(lane == 0 ? 0.f : li, pi.x));
    const float2 rr = add(splat<float2>(1.f), dr);
    const float2 dldx = fma(gr, di, mul(neg(gi), rr));  // Im(conj(gbar) r); times 2 pi later
    adj_x = add(adj_x, dldx);
    adj_tau = __fmaf_rn(dldx.x, fe.x, __fmaf_rn(dldx.y, fe.y, adj_tau));
    // the prefactor: r = rho E, so conj(gbar_rho) rho = sum conj(gbar) r, whose
    // imaginary part is the sum of dldx
    adj_rr = __fmaf_rn(gr.x, rr.x, __fmaf_rn(gr.y, rr.y, __fmaf_rn(gi.x, di.x, __fmaf_rn(gi.y, di.y, adj_rr))));
    adj_ri = __fadd_rn(adj_ri, __fadd_rn(dldx.x, dldx.y));
  }
}
}  // namespace pv

// ---------------------------------------------------------------------------
// Mixed precision.  PHASE64 = false: phase as float pairs (FP32 pipe);
// PHASE64 = true: phase accumulated in native FP64.  ND = number of
// detectors, a compile-time constant so that the independent chains of the
// detector pair and the single detector interleave in one instruction stream.
// ---------------------------------------------------------------------------
//
// FUSED: a block of at most kSetupWalkers walkers runs their set-up itself, into
// shared memory, on its first warps, while the others stage the tables; the tangents,
// which only a walker's epilogue reads, follow on the last warps (those with the
// fewest walkers) beside the other warps' slot loops.  Beside the set-up they took its
// instruction fetches: its first phase 7.5 k clocks instead of 2.5 k, the whole set-up
// 18 k (2 detectors, 777 walkers) of a launch's 25 k.  One launch, no workspace, no records through
// memory, and no gap between two kernels.  Small batches are bound by the
// host's launches and by the set-up's latency: 48 walkers, 1 detector, 100 bins, log L
// 9.6 -> 8.1 us on the GPU and 15.0 -> 11.4 us per eager call; 3 detectors, 500 bins,
// with the gradient, on the GPU: 48 walkers 13.0 -> 12.3 us, 4096 walkers 33.7 -> 33.3 us by
// the tangents' place and the staging by the other warps alone (1 detector, 100 bins,
// 4096 walkers 16.9 -> 15.7 us).  More walkers per block than lanes (kSetupWalkers) would run the
// set-up in turns while the FP32 pipe idles: those batches keep the set-up
// kernel, whose blocks overlap one another.
template <int ND, bool GRAD, bool PHASE64, bool MALA, bool FUSED>
__global__ void __launch_bounds__(kThreads)
    k_rb_mixed(typename std::conditional<FUSED, FusedArgs, LaunchArgs>::type a) {
  static_assert(!MALA || GRAD, "the MALA step needs the gradient");
  static_assert(!(FUSED && PHASE64), "the FP64-phase path has FP64 records");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const EventDev& ev = a.ev;
  constexpr int D = ND;
  const int Ep = ev.e_pad, Bp = ev.b_pad, B = ev.n_bins, E = ev.n_edges;
  const BaseRead base_read = event_base_read(ev);  // in flight across the staging

  // Stage the tables (16-byte asynchronous copies, all in flight at once).
  const float* sbin;
#ifdef RB_BOUNDS_CHECK
  unsigned smem_bytes;
  asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(smem_bytes));
  const size_t smem16 = smem_bytes / 16;
#else
  constexpr size_t smem16 = 0;  // unused
#endif
  const float4* g4 = nullptr;  // slot image: [kNBasis + 1][NS] basis values and f_e of the slots' edge pairs
  const double* g64 = nullptr;
  const double* f64 = nullptr;
  constexpr int kStageFrom = FUSED ? kDdRoleThreads : 0;  // a FUSED block's role warps leave it to the others
  {
    const int tid = (int)threadIdx.x - kStageFrom, nth = kThreads - kStageFrom;
    if (!PHASE64) {
      const float4* src = reinterpret_cast<const float4*>(ev.slot32);
      float4* dst = reinterpret_cast<float4*>(smem_raw);
      const size_t n4 = ev.slot32_floats / 4;
      if (tid >= 0)
        for (size_t i = tid; i < n4; i += nth) cp_async16(&dst[RB_IDX(i, smem16, 104)], &src[i]);
      const float* s = reinterpret_cast<const float*>(smem_raw);
      g4 = reinterpret_cast<const float4*>(s);
      sbin = s + (size_t)4 * (kNBasis + 1) * ev.n_slots;
    } else {
      const size_t n_e64 = (size_t)(kNBasis + 1) * Ep;  // g[10][Ep], f[Ep]
      const double2* src = reinterpret_cast<const double2*>(ev.tab64);
      double2* dst = reinterpret_cast<double2*>(smem_raw);
      for (size_t i = tid; i < n_e64 / 2; i += nth) cp_async16(&dst[RB_IDX(i, smem16, 104)], &src[i]);
      const size_t nb = ev.tab32_floats - ev.edge32_floats;
      const float4* bsrc = reinterpret_cast<const float4*>(ev.tab32 + ev.edge32_floats);
      float4* bdst = reinterpret_cast<float4*>(smem_raw + n_e64 * sizeof(double));
      for (size_t i = tid; i < nb / 4; i += nth) cp_async16(&bdst[RB_IDX(i, smem16 - n_e64 / 2, 104)], &bsrc[i]);
      g64 = reinterpret_cast<const double*>(smem_raw);
      f64 = g64 + (size_t)kNBasis * Ep;
      sbin = reinterpret_cast<const float*>(smem_raw + n_e64 * sizeof(double));
    }
  }
  cp_async_commit();

  const int lane = threadIdx.x & 31;
  WarpSlot* slot = nullptr;       // this warp's slot, after the tables
  FusedRecords* fused = nullptr;  // FUSED: the block's records
  WarpWork* work;
  {
    const size_t tab_bytes = !PHASE64 ? ev.slot32_floats * sizeof(float)
                                      : (size_t)(kNBasis + 1) * Ep * sizeof(double) +
                                            (ev.tab32_floats - ev.edge32_floats) * sizeof(float);
    if constexpr (FUSED) {
      fused = reinterpret_cast<FusedRecords*>(smem_raw + tab_bytes);
      work = reinterpret_cast<WarpWork*>(smem_raw + tab_bytes + sizeof(FusedRecords)) + (threadIdx.x >> 5);
    } else {
      slot = reinterpret_cast<WarpSlot*>(smem_raw + tab_bytes) + (threadIdx.x >> 5);
      work = &slot->work;
    }
  }
  // detectors 0 and 1 form a pair when D >= 2; an odd detector count leaves
  // detector D - 1 single (bin table layout in EventDev)
  constexpr bool paired = D >= 2;
  constexpr int ds = (D & 1) ? D - 1 : -1;
  constexpr int dss = ds < 0 ? 0 : ds;
  const float4* binP = reinterpret_cast<const float4*>(sbin);                                // [3][Bp]
  const float4* binS4 = reinterpret_cast<const float4*>(sbin + (paired ? 12 * Bp : 0));      // [Bp]
  const float2* binS2 = reinterpret_cast<const float2*>(sbin + (paired ? 12 * Bp : 0) + 4 * Bp);  // [Bp]
  // each block takes a contiguous, equal share of the walkers (so every SM
  // gets W / grid of them, +-1), its warps take them in turn
  const int64_t per_blk = a.W / gridDim.x, rem_blk = a.W % gridDim.x;
  const int64_t w_begin = (int64_t)blockIdx.x * per_blk + min((int64_t)blockIdx.x, rem_blk);
  const int64_t w_end = w_begin + per_blk + ((int64_t)blockIdx.x < rem_blk ? 1 : 0);
  const int64_t warp0 = w_begin + (threadIdx.x >> 5);
  const int64_t nwarps = blockDim.x >> 5;
  const unsigned char* rec_g = static_cast<const unsigned char*>(a.ws);
  const unsigned char* tan_g = static_cast<const unsigned char*>(a.tan);
  const MalaBlock* chains = nullptr;  // FUSED MALA: the block's chains
  constexpr int kFusedTanWarps = 3 + D;
  // FUSED: theta of the block's walkers, the first and the end of its rows
  const double* theta = nullptr;
  int64_t t_begin = w_begin, t_end = w_end;
  if constexpr (FUSED) {
    theta = a.theta;
    DdSmem& S = *reinterpret_cast<DdSmem*>(fused + 1);
    if constexpr (MALA) {
      MalaBlock* mb = reinterpret_cast<MalaBlock*>(reinterpret_cast<unsigned char*>(fused) + kFusedBytes);
      mala_propose_block(a.mala, w_begin, (int)(w_end - w_begin), *mb);
      chains = mb;
      theta = &mb->theta[0][0];
      t_begin = 0;
      t_end = w_end - w_begin;
    }
    if (GRAD && threadIdx.x == kDdRoleThreads) mbar_init(&fused->tan_done, kFusedTanWarps);
    if (threadIdx.x < kDdRoleThreads) {
      setup_load_dd<true>(theta, t_begin, t_end, S);
      setup_absolute_dd(a.ec, S);
      setup_record_dd(ev.ref->dd, a.ec, S, &fused->rec[lane], w_begin + lane < w_end);
    }
  }
  // the first walker's record and tangents travel with the tables
  if (!FUSED && warp0 < w_end)
    prefetch_walker<GRAD, PHASE64>(slot, 0, PHASE64 ? nullptr : rec_g + sizeof(WalkerMixed) * RB_IDX(warp0, a.W, 101),
                                   GRAD ? tan_g + sizeof(WalkerTan<float>) * RB_IDX(warp0, a.W, 107) : nullptr, lane);
  cp_async_wait_all();
  __syncthreads();
  if constexpr (FUSED && GRAD) {
    const int which = (int)(threadIdx.x >> 5) - (kThreads / 32 - kFusedTanWarps);
    if (which >= 0) {
      tangent_warp<float>(theta, t_end, t_begin, a.ec, fused->tan, which);
      __syncwarp();
      if (lane == 0) mbar_arrive(&fused->tan_done);
    }
  }
  const double base_logl = event_base_value(ev, base_read);

  // the bound on |g_k| or f that this lane's phase term takes (the record
  // expansion below: lane k < kNBasis basis k, lane kNBasis + 3 d detector d's
  // delay), read once into the warp's slot: indexed by lane, a constant-bank
  // load serialises
  if (!PHASE64) {
    const int j = lane - kNBasis;
    const int gk = lane < kNBasis ? lane : (j < 3 * D && j % 3 == 0 ? kNBasis : -1);
    work->lane_gmax[lane] = gk >= 0 ? ev.gmax[gk] : 0.f;
  }

  // the MALA step of walker w, its log L and gradient (lane j: component j) at hand
  auto mala_step = [&](int64_t w, double logl, double gth) {
    if constexpr (FUSED) {
      const int l = (int)(w - w_begin);
      const MalaWalker mw{chains->inside[l] != 0, chains->lu[l], chains->jac9[l], chains->jac12[l],
                          lane == 9 ? chains->zp9[l] : lane == 12 ? chains->zp12[l] : lane < kNPar ? chains->theta[l][lane] : 0.0};
      mala_finish(a.mala, w, lane, logl, gth, mw);
    } else {
      mala_finish(a.mala, w, lane, logl, gth, mala_walker(a.mala, w, lane));
    }
  };
  int buf = 0;
  for (int64_t w = warp0; w < w_end; w += nwarps, buf ^= 1) {
    if (!FUSED) cp_async_wait_all();  // this walker's record and tangents
    __syncwarp();  // ... visible to the warp; the previous walker's reads of wc and of buffer buf ^ 1 done
    // ---- per-walker constants (uniform across the warp), in shared memory ----
    const int64_t wl = FUSED ? RB_IDX(w - w_begin, kSetupWalkers, 101) : 0;
    WalkerMixed& rec = FUSED ? fused->rec[wl] : slot->rec[buf];
    float4* const wc = rec.q;
    double dc64[kNBasis];
    double tau64[kMaxDet];
    pv::DetState<float2> P;  // detectors 0, 1: accumulators (constants come from wc)
    pv::DetState<float> S;   // detector ds
    int valid;
    unsigned walker_ex = 0;  // float-float path: exponent field of the walker's phase-term bound
    if (!PHASE64) {
      valid = rec.valid;
#pragma unroll
      for (int k = 0; k < kNBasis; ++k) dc64[k] = 0.0;
#pragma unroll
      for (int d = 0; d < kMaxDet; ++d) tau64[d] = 0.0;
      // each constant in both halves of a pair (the slot loop's operands):
      // lane k < kNBasis takes dc_k, lane kNBasis + 3 d + m the delay (m = 0),
      // prefactor ratio (1) or its difference from 1 (2) of detector d
      float mag = 0.f;  // the lane's bound on |its phase term| [turns]
      if (lane < kNBasis + 3 * D) {
        const float* f = reinterpret_cast<const float*>(wc);
        int iu, iv;
        if (lane < kNBasis) {
          iu = wm_dc_hi(lane);
          iv = wm_dc_lo(lane);
        } else {
          const int j = lane - kNBasis, d = j / 3, m = j - 3 * d;
          if (d == ds) {
            iu = kWmSingle + (m == 0 ? 0 : 2 + 2 * m);
          } else {
            iu = (m == 0 ? kWmTauPair : (m == 1 ? kWmRhoPair : kWmSigPair)) + d;
          }
          iv = iu + (d == ds ? 1 : 2);
        }
        const float u = f[iu], v = f[iv];
        work->dup[lane] = make_float4(u, u, v, v);
        mag = fabsf(u) * work->lane_gmax[lane];
      }
      // the walker's rounding constant m = 1.5 * 2^23 q with q = 2^-20 of a
      // power of two above every phase term (at least 2^-62 turns): then each
      // product's high part is below 2^22 q, and the eleven of a detector's
      // phase (ten basis terms and the delay) add to less than 2^24 q
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mag = fmaxf(mag, __shfl_xor_sync(0xffffffffu, mag, o));
      const unsigned ex = min(max((__float_as_uint(mag) >> 23) & 0xffu, 64u), 250u);  // mag < 2^(ex - 126)
      walker_ex = ex;
      if (lane == 0) {
        const float m = __uint_as_float(((ex + 4u) << 23) | 0x400000u);  // 1.5 * 2^(ex - 123)
        work->dup[kNBasis + 3 * kMaxDet] = make_float4(m, m, m, m);
      }
    } else {
      float rho[kMaxDet][2], sg[kMaxDet][2];
      const WalkerF64* s = reinterpret_cast<const WalkerF64*>(a.ws) + w;
      valid = s->valid;
#pragma unroll
      for (int k = 0; k < kNBasis; ++k) dc64[k] = s->dc[k];
#pragma unroll
      for (int d = 0; d < kMaxDet; ++d) {
        tau64[d] = s->tau[d];
        rho[d][0] = (float)s->rho[d][0]; rho[d][1] = (float)s->rho[d][1];
        sg[d][0] = (float)s->sig[d][0]; sg[d][1] = (float)s->sig[d][1];
      }
      __syncwarp();  // the previous walker's reads of this buffer are done
      if (lane == 0) {
        // the phase and delay quads are not read on this path
#pragma unroll
        for (int q = 0; q < 6; ++q) wc[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        wc[6] = make_float4(rho[0][0], rho[1][0], rho[0][1], rho[1][1]);
        wc[7] = make_float4(sg[0][0], sg[1][0], sg[0][1], sg[1][1]);
        wc[8] = make_float4(0.f, 0.f, 0.f, 0.f);
        wc[9] = make_float4(rho[dss][0], rho[dss][1], sg[dss][0], sg[dss][1]);
      }
    }
    __syncwarp();
    if (!FUSED) {
      // the next walker's record and tangents, into the other buffer (issued
      // after this walker's shared-memory reads above)
      const int64_t wn = w + nwarps;
      if (wn < w_end)
        prefetch_walker<GRAD, PHASE64>(slot, buf ^ 1, PHASE64 ? nullptr : rec_g + sizeof(WalkerMixed) * RB_IDX(wn, a.W, 101),
                                       GRAD ? tan_g + sizeof(WalkerTan<float>) * RB_IDX(wn, a.W, 107) : nullptr, lane);
    }
    if (!valid) {
      if constexpr (MALA) {
        mala_step(w, -INFINITY, 0.0);
      } else {
        if (lane == 0) a.logl[w] = -INFINITY;
        if (GRAD && lane < kNPar) a.grad[w * kNPar + lane] = 0.0;
      }
      continue;
    }
    if (!PHASE64 && walker_ex > 126u + 18u) {
      // a phase term beyond 2^18 turns (~1.6e6 rad): past the range of the
      // float-pair phase sums' whole-turn reductions; not evaluated (NaN,
      // rejected by the MALA step)
      if constexpr (MALA) {
        mala_step(w, -INFINITY, 0.0);
      } else {
        if (lane == 0) a.logl[w] = __longlong_as_double(0x7ff8000000000000ll);
        if (GRAD && lane < kNPar) a.grad[w * kNPar + lane] = __longlong_as_double(0x7ff8000000000000ll);
      }
      continue;
    }

    // float-pair accumulators: for walkers far from the fiducial point the
    // per-bin terms add up to about -log L(theta_ref), so a single float would
    // lose ~1e-3 of absolute precision
    constexpr int kNV = kNBasis + 3 * D;
    float lh, ll;   // the lane's share of log L - log L(theta_ref), a float pair
    float v[kNV];   // the lane's adjoint sums: basis coefficients, then per detector the delay and the ratio re/im
    if constexpr (!PHASE64) {
      // slot loop: both halves of every paired value are edges of this walker
      const int NS = ev.n_slots;
      const float4* const wd = work->dup;
      float2 acc = make_float2(0.f, 0.f), acc_lo = acc;
      // the adjoint sums of a lane's two edges in one float each (as pairs,
      // the extra registers spilled)
      float adj_c[kNBasis];
      float adj_tau[D], adj_rr[D], adj_ri[D];
#pragma unroll
      for (int k = 0; k < kNBasis; ++k) adj_c[k] = 0.f;
#pragma unroll
      for (int d = 0; d < D; ++d) adj_tau[d] = adj_rr[d] = adj_ri[d] = 0.f;
      // walkers whose phase terms reach beyond 2^12 turns take a second
      // whole-turn reduction of the phase (the low sum can then carry it past
      // the half-angle polynomials' range): a second copy of the loop, so
      // that the others pay nothing for it
      auto slot_loop = [&](auto wide_c) {
      constexpr bool WIDE = decltype(wide_c)::value;
      for (int s0 = 0; s0 < NS; s0 += 32) {
        const int sl = RB_IDX(s0 + lane, NS, 102);
        // detector-independent phase sum_k dc_k g_k(f_e) / 2pi [turns] of the
        // two edges, as an exact sum of multiples of the walker's q (sh) and a
        // small remainder (sl_lo)
        const float4 mq = lds4(wd + kNBasis + 3 * kMaxDet);
        const float2 m2 = make_float2(mq.x, mq.y);
        float2 sh = make_float2(0.f, 0.f), sl_lo = sh;
#pragma unroll
        for (int k = 0; k < kNBasis; ++k) {
          const float4 g = g4[k * NS + sl];  // {g_hi(e_A), g_hi(e_B), g_lo(e_A), g_lo(e_B)}
          const float4 c = lds4(wd + k);     // {dc_hi, dc_hi, dc_lo, dc_lo}
          pv::split_acc(make_float2(c.x, c.y), make_float2(c.z, c.w), make_float2(g.x, g.y), make_float2(g.z, g.w), m2, sh,
                        sl_lo);
        }
        const float4 f4 = g4[kNBasis * NS + sl];
        const float2 fe = make_float2(f4.x, f4.y), fe_lo = make_float2(f4.z, f4.w);
        float2 vsum = make_float2(0.f, 0.f), adj_x = vsum;
#pragma unroll
        for (int d = 0; d < D; ++d) {
          const float4 tt = lds4(wd + kNBasis + 3 * d);
          float2 yh = sh, yl = sl_lo;
          pv::split_acc(make_float2(tt.x, tt.y), make_float2(tt.z, tt.w), fe, fe_lo, m2, yh, yl);
          float2 y = pv::frac(yh, yl);
          if constexpr (WIDE) y = pv::frac1(y);
          const float4* sb = reinterpret_cast<const float4*>(sbin + (size_t)d * kSlotBinFloats * NS);
          const float4 q0 = sb[sl], q1 = sb[NS + sl], q2 = sb[2 * NS + sl];
          const float2 bt[6] = {make_float2(q0.x, q0.y), make_float2(q0.z, q0.w), make_float2(q1.x, q1.y),
                                make_float2(q1.z, q1.w), make_float2(q2.x, q2.y), make_float2(q2.z, q2.w)};
          pv::det_edge_slot<GRAD>(y, lds4(wd + kNBasis + 3 * d + 1), lds4(wd + kNBasis + 3 * d + 2), bt, lane, fe, vsum,
                                  adj_x, adj_tau[d], adj_rr[d], adj_ri[d]);
        }
        pv::add_acc(acc, acc_lo, vsum);
        if (GRAD) {
          // the high halves only: 8-byte loads (shared-memory bandwidth is
          // about as busy as the FMA pipe in this loop)
          const float2* g2 = reinterpret_cast<const float2*>(g4);
#pragma unroll
          for (int k = 0; k < kNBasis; ++k) {
            const float2 g = g2[2 * (k * NS + sl)];
            adj_c[k] = __fmaf_rn(adj_x.x, g.x, __fmaf_rn(adj_x.y, g.y, adj_c[k]));
          }
        }
      }
      };
      if (walker_ex > 126u + 12u) slot_loop(std::true_type{});
      else slot_loop(std::false_type{});
      lh = acc.x;
      ll = acc_lo.x;
      ff_add(lh, ll, acc.y, acc_lo.y);
#pragma unroll
      for (int k = 0; k < kNBasis; ++k) v[k] = adj_c[k];
#pragma unroll
      for (int d = 0; d < D; ++d) {
        v[kNBasis + d] = adj_tau[d];
        v[kNBasis + D + d] = adj_rr[d];
        v[kNBasis + 2 * D + d] = adj_ri[d];
      }
    } else {
      // FP64 phase: one edge per lane, lane l of chunk c at edge 31 c + l
      P.acc = P.acc_lo = P.adj_tau = P.adj_rr = P.adj_ri = make_float2(0.f, 0.f);
      S.acc = S.acc_lo = S.adj_tau = S.adj_rr = S.adj_ri = 0.f;
      float2 adj_c[kNBasis / 2];
#pragma unroll
      for (int q = 0; q < kNBasis / 2; ++q) adj_c[q] = make_float2(0.f, 0.f);

      for (int c0 = 0; c0 < B; c0 += 31) {
        const int e = c0 + lane;
        const bool has_edge = e < E;
        const bool has_bin = (lane < 31) && (e < B);
        const int ee = RB_IDX(has_edge ? e : E - 1, Ep, 102);
        const int eb = RB_IDX(has_bin ? e : 0, Bp, 103);
        double x64 = 0.0;
#pragma unroll
        for (int k = 0; k < kNBasis; ++k) x64 = ::fma(dc64[k], g64[k * Ep + ee], x64);
        const float fe = (float)f64[ee];

        float adj_x = 0.f;
        if constexpr (paired) {
          const float4 rr = lds4(wc + 6), ss = lds4(wc + 7);
          P.rho_r = make_float2(rr.x, rr.y); P.rho_i = make_float2(rr.z, rr.w);
          P.sig_r = make_float2(ss.x, ss.y); P.sig_i = make_float2(ss.z, ss.w);
          const double x0 = ::fma(f64[ee], tau64[0], x64), x1 = ::fma(f64[ee], tau64[1], x64);
          const float2 y = make_float2((float)(x0 - rint(x0)), (float)(x1 - rint(x1)));
          const float4 q0 = binP[eb], q1 = binP[Bp + eb], q2 = binP[2 * Bp + eb];
          const float2 bt[6] = {make_float2(q0.x, q0.y), make_float2(q0.z, q0.w), make_float2(q1.x, q1.y),
                                make_float2(q1.z, q1.w), make_float2(q2.x, q2.y), make_float2(q2.z, q2.w)};
          const float2 g = pv::det_edge<GRAD>(y, P, bt, has_bin, has_edge, lane, make_float2(fe, fe));
          adj_x = __fadd_rn(g.x, g.y);
        }
        if constexpr (ds >= 0) {
          const float4 rs = lds4(wc + 9);
          S.rho_r = rs.x; S.rho_i = rs.y; S.sig_r = rs.z; S.sig_i = rs.w;
          const double xd = ::fma(f64[ee], tau64[ds], x64);
          const float y = (float)(xd - rint(xd));
          const float4 q0 = binS4[eb];
          const float2 q1 = binS2[eb];
          const float bt[6] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y};
          adj_x = __fadd_rn(adj_x, pv::det_edge<GRAD>(y, S, bt, has_bin, has_edge, lane, fe));
        }
        if (GRAD && has_edge) {
          const float2 ax = make_float2(adj_x, adj_x);
#pragma unroll
          for (int q = 0; q < kNBasis / 2; ++q)
            adj_c[q] = pv::fma(ax, make_float2((float)g64[2 * q * Ep + ee], (float)g64[(2 * q + 1) * Ep + ee]),
                               adj_c[q]);
        }
      }
      lh = S.acc;
      ll = S.acc_lo;
      if constexpr (paired) {
        ff_add(lh, ll, P.acc.x, P.acc_lo.x);
        ff_add(lh, ll, P.acc.y, P.acc_lo.y);
      }
#pragma unroll
      for (int q = 0; q < kNBasis / 2; ++q) {
        v[2 * q] = adj_c[q].x;
        v[2 * q + 1] = adj_c[q].y;
      }
      if constexpr (paired) {
        v[kNBasis + 0] = P.adj_tau.x;
        v[kNBasis + 1] = P.adj_tau.y;
        v[kNBasis + D + 0] = P.adj_rr.x;
        v[kNBasis + D + 1] = P.adj_rr.y;
        v[kNBasis + 2 * D + 0] = P.adj_ri.x;
        v[kNBasis + 2 * D + 1] = P.adj_ri.y;
      }
      if constexpr (ds >= 0) {
        v[kNBasis + ds] = S.adj_tau;
        v[kNBasis + D + ds] = S.adj_rr;
        v[kNBasis + 2 * D + ds] = S.adj_ri;
      }
    }

    // the walker's sum as a float pair (FP32 pipe); FP64 only for the result
    warp_sum_ff(lh, ll);
    const double logl = base_logl + (f2d_int(lh) + f2d_int(ll));
    if (!MALA && lane == 0) a.logl[RB_IDX(w, a.W, 105)] = logl;
    if (GRAD) {
      const float two_pi = 6.28318530717958648f;
      // the walker's adjoint sums (basis coefficients, then per detector the
      // delay and the prefactor ratio re/im) by one transposed warp sum
      warp_transposed_sums(v, lane, work->red);
      __syncwarp();
      float ac[kNBasis], at[kMaxDet], ar[kMaxDet][2];
#pragma unroll
      for (int k = 0; k < kNBasis; ++k) ac[k] = two_pi * work->red[k];
#pragma unroll
      for (int d = 0; d < kMaxDet; ++d) {
        at[d] = d < D ? two_pi * work->red[kNBasis + d] : 0.f;
        ar[d][0] = d < D ? work->red[kNBasis + D + d] : 0.f;
        ar[d][1] = d < D ? work->red[kNBasis + 2 * D + d] : 0.f;
      }
      if constexpr (PHASE64) {
        // this path sums gbar conj(E) = gbar_rho: G_d = conj(gbar_rho) rho
        float rho[kMaxDet][2];
        const float4 r01 = lds4(wc + 6), rs = lds4(wc + 9);
        rho[0][0] = r01.x; rho[1][0] = r01.y; rho[0][1] = r01.z; rho[1][1] = r01.w;
        if (ds >= 0) { rho[dss][0] = rs.x; rho[dss][1] = rs.y; }
        if (D < kMaxDet) rho[kMaxDet - 1][0] = rho[kMaxDet - 1][1] = 0.f;
#pragma unroll
        for (int d = 0; d < kMaxDet; ++d) {
          const float a_r = ar[d][0], a_i = ar[d][1];
          ar[d][0] = a_r * rho[d][0] + a_i * rho[d][1];
          ar[d][1] = a_r * rho[d][1] - a_i * rho[d][0];
        }
      }
      double g = 0.0;
      bool tan_ok = true;
      if constexpr (FUSED) tan_ok = mbar_wait(&fused->tan_done);
      if (lane < kNPar) {
        const WalkerTan<float>& tn = FUSED ? fused->tan[wl] : *reinterpret_cast<const WalkerTan<float>*>(slot->tan[buf]);
        g = tan_ok ? f2d_int(chain_rule_lanes<D>(lane, ac, at, ar, tn)) : __longlong_as_double(0x7ff8000000000000ll);
      }
      if constexpr (MALA) mala_step(w, logl, g);
      else if (lane < kNPar) a.grad[RB_IDX(w * kNPar + lane, a.W * kNPar, 106)] = g;
    }
  }
}

// ---------------------------------------------------------------------------
// Plain FP64 comparison path: lane l of chunk c at edge 31 c + l, everything in
// FP64, tables read through the cache from global memory.
//
// Bound: the FP64 pipe (one warp instruction per ~65 clocks per SM
// sub-partition, whatever the lanes), so what counts is FP64 instructions per
// edge: with three detectors 170 -- the bin term in the coefficients of its edge
// values (as det_edge_slot; the beta1 term, zero for a ratio of constant
// modulus, left out), e^{-2 pi i x} - 1 from one quarter-turn reduction, the
// prefactor's adjoint as the sum of conj(gbar) r -- and 21 additions for the warp
// sums of 20 values (transposed).  In the general form (alpha0, alpha1,
// beta0, beta1, sincospi, butterflies) it was 251 and 100.  1000 walkers, 200
// bins: 150 -> 79 us (FP64 pipe 84 -> 89 % busy), errors against the oracle unchanged.
// ---------------------------------------------------------------------------
// e with |x| < 2^(e + 1) (inf and NaN: the largest).
__device__ __forceinline__ int exponent64(double x) { return ((__double2hiint(x) >> 20) & 0x7ff) - 1023; }
__device__ __forceinline__ int exponent32(float x) { return ((__float_as_int(x) >> 23) & 0xff) - 127; }

template <int ND, bool GRAD, bool MALA = false>
__global__ void __launch_bounds__(256) k_rb_f64(LaunchArgs a) {
  static_assert(!MALA || GRAD, "the MALA step needs the gradient");
  constexpr int kNV = 1 + (GRAD ? kNBasis + 3 * ND : 0);  // log L; basis coefficients, delays, G re, G im
  __shared__ double s_red[256 / 32][32];
  const EventDev& ev = a.ev;
  const int Ep = ev.e_pad, Bp = ev.b_pad, B = ev.n_bins, E = ev.n_edges;
  const double* __restrict__ g64 = ev.tab64;
  const double* __restrict__ f64 = ev.tab64 + (size_t)kNBasis * Ep;
  const double* __restrict__ bin64 = ev.tab64 + (size_t)(kNBasis + 1) * Ep;
  const int lane = threadIdx.x & 31;
  double* red = s_red[threadIdx.x >> 5];
  // each block takes a contiguous, equal share of the walkers (so every SM
  // gets W / grid of them, +-1), its warps take them in turn
  const int64_t per_blk = a.W / gridDim.x, rem_blk = a.W % gridDim.x;
  const int64_t w_begin = (int64_t)blockIdx.x * per_blk + min((int64_t)blockIdx.x, rem_blk);
  const int64_t w_end = w_begin + per_blk + ((int64_t)blockIdx.x < rem_blk ? 1 : 0);
  const int64_t warp0 = w_begin + (threadIdx.x >> 5);
  const int64_t nwarps = blockDim.x >> 5;
  const double base_logl = event_base_logl(ev);
  for (int64_t w = warp0; w < w_end; w += nwarps) {
    const WalkerF64* s = reinterpret_cast<const WalkerF64*>(a.ws) + w;
    if (!s->valid) {
      if (MALA) {
        mala_finish(a.mala, w, lane, -INFINITY, 0.0, mala_walker(a.mala, w, lane));
      } else {
        if (lane == 0) a.logl[w] = -INFINITY;
        if (GRAD && lane < kNPar) a.grad[w * kNPar + lane] = 0.0;
      }
      continue;
    }
    double dc[kNBasis], tau[ND], rho[ND][2], sig[ND][2];
#pragma unroll
    for (int k = 0; k < kNBasis; ++k) dc[k] = s->dc[k];
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      tau[d] = s->tau[d];
      rho[d][0] = s->rho[d][0]; rho[d][1] = s->rho[d][1];
      sig[d][0] = s->sig[d][0]; sig[d][1] = s->sig[d][1];
    }
    double v[kNV];
#pragma unroll
    for (int i = 0; i < kNV; ++i) v[i] = 0.0;
    // a walker whose phase may reach 2^49 turns (a delay of 1e12 s, say) loses the whole
    // turns of its phases before the quarter-turn reduction.  From the exponents of its terms
    // c_k g_k and f tau, on the integer pipe: eleven terms below 2^(m + 2) each
    int m = -4096;
#pragma unroll
    for (int k = 0; k < kNBasis; ++k) m = max(m, exponent64(dc[k]) + exponent32(ev.gmax[k]));
#pragma unroll
    for (int d = 0; d < ND; ++d) m = max(m, exponent64(tau[d]) + exponent32(ev.gmax[kNBasis]));
    // (as a second copy of the loop: one with the test inside took 98.9 us for 96.3)
    auto edges = [&](auto far_c) {
      for (int c0 = 0; c0 < B; c0 += 31) {
        const int e = c0 + lane;
        const bool has_edge = e < E;
        const bool has_bin = (lane < 31) && (e < B);
        const int ee = has_edge ? e : E - 1, eb = has_bin ? e : 0;
        double x = 0.0;
  #pragma unroll
        for (int k = 0; k < kNBasis; ++k) x = fma(dc[k], g64[k * Ep + ee], x);
        const double fe = f64[ee];
        double adj_x = 0.0;
  #pragma unroll
        for (int d = 0; d < ND; ++d) {
          double em_r, em_i;
          double y = fma(fe, tau[d], x);
          if constexpr (decltype(far_c)::value) y -= rint(y);
          expm1_neg_turns64(y, em_r, em_i);
          const double dr = fma(rho[d][0], em_r, fma(-rho[d][1], em_i, sig[d][0]));
          const double di = fma(rho[d][0], em_i, fma(rho[d][1], em_r, sig[d][1]));
          const double nr = __shfl_down_sync(kFull, dr, 1);
          const double ni = __shfl_down_sync(kFull, di, 1);
          // the bin on the edge's right; zero coefficients where there is none
          const double* bt = bin64 + (size_t)d * 6 * Bp + eb;
          const double gmr = has_bin ? bt[0] : 0.0, gpr = has_bin ? bt[Bp] : 0.0, gmi = has_bin ? bt[2 * Bp] : 0.0;
          const double gpi = has_bin ? bt[3 * Bp] : 0.0, q = has_bin ? bt[5 * Bp] : 0.0;
          const double sr = dr + nr, si = di + ni;
          v[0] = fma(gmr, dr, v[0]);
          v[0] = fma(gpr, nr, v[0]);
          v[0] = fma(gmi, di, v[0]);
          v[0] = fma(gpi, ni, v[0]);
          v[0] = fma(q, fma(sr, sr, si * si), v[0]);
          if (GRAD) {
            const double h = has_bin ? bt[4 * Bp] : 0.0;
            double gr = fma(h, sr, gmr), gi = fma(h, si, gmi);
            const double lr = __shfl_up_sync(kFull, fma(h, sr, gpr), 1), li = __shfl_up_sync(kFull, fma(h, si, gpi), 1);
            gr += lane > 0 ? lr : 0.0;
            gi += lane > 0 ? li : 0.0;
            if (has_edge) {
              const double rr = 1.0 + dr;
              const double dldx = fma(gr, di, -(gi * rr));  // Im(conj(gbar) r)
              adj_x += dldx;
              v[1 + kNBasis + d] = fma(dldx, fe, v[1 + kNBasis + d]);
              v[1 + kNBasis + ND + d] = fma(gr, rr, fma(gi, di, v[1 + kNBasis + ND + d]));
              v[1 + kNBasis + 2 * ND + d] += dldx;
            }
          }
        }
        if (GRAD && has_edge) {
  #pragma unroll
          for (int k = 0; k < kNBasis; ++k) v[1 + k] = fma(adj_x, g64[k * Ep + ee], v[1 + k]);
        }
      }
    };
    if (m < 49 - 6) edges(std::false_type{});
    else edges(std::true_type{});
    warp_transposed_sums(v, lane, red);
    __syncwarp();
    const double logl = base_logl + red[0];
    if (!MALA && lane == 0) a.logl[RB_IDX(w, a.W, 105)] = logl;
    if (GRAD) {
      double ac[kNBasis], at[ND], G[ND][2];
#pragma unroll
      for (int k = 0; k < kNBasis; ++k) ac[k] = kTwoPi * red[1 + k];
#pragma unroll
      for (int d = 0; d < ND; ++d) {
        at[d] = kTwoPi * red[1 + kNBasis + d];
        G[d][0] = red[1 + kNBasis + ND + d];
        G[d][1] = red[1 + kNBasis + 2 * ND + d];
      }
      double g = 0.0;
      if (lane < kNPar) g = chain_rule_lanes<ND>(lane, ac, at, G, reinterpret_cast<const WalkerTan<double>*>(a.tan)[w]);
      if (MALA) mala_finish(a.mala, w, lane, logl, g, mala_walker(a.mala, w, lane));
      else if (lane < kNPar) a.grad[RB_IDX(w * kNPar + lane, a.W * kNPar, 106)] = g;
    }
    __syncwarp();  // red is read before the next walker's sums
  }
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
size_t mixed_smem_slot_bytes() { return (size_t)(kThreads / 32) * sizeof(WarpSlot); }

size_t mixed_smem_bytes(const EventDev& ev, bool phase64) {
  const size_t wc = (size_t)(kThreads / 32) * sizeof(WarpSlot);
  if (!phase64) return ev.slot32_floats * sizeof(float) + wc;
  return (size_t)(kNBasis + 1) * ev.e_pad * sizeof(double) + (ev.tab32_floats - ev.edge32_floats) * sizeof(float) + wc;
}

// Occupancy per (kernel, shared-memory size), cached in a fixed table (no
// heap allocation on the launch path): the query costs host time otherwise.
struct OccEntry {
  const void* fn;
  size_t smem;
  int blocks;
};
constexpr int kOccSlots = 256;
static std::mutex g_occ_mu;
static OccEntry g_occ[kOccSlots];
static int g_occ_n = 0;
constexpr int kSmemRaised = 64;
static const void* g_smem_raised[kSmemRaised];
static int g_smem_raised_n = 0;

static size_t smem_optin_max() {
  static std::once_flag once;
  static int n = 0;
  std::call_once(once, [] {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
      n = 0;
  });
  return (size_t)n;
}

static cudaError_t blocks_per_sm(const void* fn, int threads, size_t smem, int* out) {
  std::lock_guard<std::mutex> lk(g_occ_mu);
  for (int i = 0; i < g_occ_n; ++i)
    if (g_occ[i].fn == fn && g_occ[i].smem == smem) {
      *out = g_occ[i].blocks;
      return cudaSuccess;
    }
  cudaError_t err = cudaSuccess;
  bool raised = false;
  for (int i = 0; i < g_smem_raised_n; ++i) raised = raised || g_smem_raised[i] == fn;
  if (!raised) {
    // allow any dynamic shared-memory size up to the device limit (less the
    // kernel's static shared memory) once, so that launches for different
    // events never shrink it for one another
    int dev = 0, smem_max = 0;
    cudaFuncAttributes fa{};
    err = cudaGetDevice(&dev);
    if (err == cudaSuccess) err = cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (err == cudaSuccess) err = cudaFuncGetAttributes(&fa, fn);
    if (err == cudaSuccess)
      err = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max - (int)fa.sharedSizeBytes);
    if (err != cudaSuccess) return err;
    if (g_smem_raised_n < kSmemRaised) g_smem_raised[g_smem_raised_n++] = fn;
  }
  int n = 0;
  err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, threads, smem);
  if (err != cudaSuccess) return err;
  if (g_occ_n < kOccSlots) g_occ[g_occ_n++] = OccEntry{fn, smem, n};
  *out = n;
  return cudaSuccess;
}

constexpr int64_t kThinWalkers = 4;  // an SM's sub-partitions

// Blocks of a batch of W walkers, at most n_max.  spread: a batch that does not
// fill the SMs with 16 walkers per block takes more of them, down to one walker
// per SM sub-partition (the warps of a block share its FP32 pipe; below four
// walkers nothing is left to share).  Otherwise (launches that share the GPU with
// others: the server's, RB_SHARED) the blocks stay dense: fewer SMs are held, for
// longer.  A call of 1024 walkers with the gradient, 3 detectors, 500 bins, one after
// the other on one stream: spread (and in one launch with the set-up, see FUSED) 18.4
// us, dense 24.7; on eight branches of a graph: 15.6 and 7.9.  (64 walkers: 12.3 and
// 25.0; 2.1 and 3.5.)
static int64_t mixed_grid(int64_t W, bool spread, int n_sm, int64_t n_max) {
  const int64_t dense = (W * 32 + kThreads - 1) / kThreads;
  const int64_t thin = spread ? std::min<int64_t>((W + kThinWalkers - 1) / kThinWalkers, n_sm) : 0;
  return std::min<int64_t>(std::max<int64_t>(dense, thin), n_max);
}

template <int ND, bool GRAD, bool PHASE64, bool MALA>
static cudaError_t launch_mixed_nd(const LaunchArgs& a, bool spread, cudaStream_t s, int n_sm) {
  // the kernel copies records in 16-byte and tangents in 8-byte asynchronous copies
  if (reinterpret_cast<uintptr_t>(a.ws) % 16 != 0 || (GRAD && reinterpret_cast<uintptr_t>(a.tan) % 8 != 0))
    return cudaErrorMisalignedAddress;
  const size_t smem = mixed_smem_bytes(a.ev, PHASE64);
  auto* fn = k_rb_mixed<ND, GRAD, PHASE64, MALA, false>;
  int per_sm = 0;
  cudaError_t err = blocks_per_sm(reinterpret_cast<const void*>(fn), kThreads, smem, &per_sm);
  if (err != cudaSuccess) return err;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  fn<<<(unsigned)mixed_grid(a.W, spread, n_sm, (int64_t)per_sm * n_sm), kThreads, smem, s>>>(a);
  return cudaGetLastError();
}

template <bool GRAD, bool PHASE64, bool MALA = false>
static cudaError_t launch_mixed_t(const LaunchArgs& a, bool spread, cudaStream_t s, int n_sm) {
  switch (a.ev.n_det) {
    case 1: return launch_mixed_nd<1, GRAD, PHASE64, MALA>(a, spread, s, n_sm);
    case 2: return launch_mixed_nd<2, GRAD, PHASE64, MALA>(a, spread, s, n_sm);
    case 3: return launch_mixed_nd<3, GRAD, PHASE64, MALA>(a, spread, s, n_sm);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_rb_mixed(const EventDev& ev, const void* ws, const void* tan, int64_t W, double* logl, double* grad,
                            bool phase64, bool spread, cudaStream_t s, int n_sm, const MalaArgs* mala) {
  LaunchArgs a{ev, ws, tan, W, logl, grad, {}};
  if (mala) {
    a.mala = *mala;
    return phase64 ? launch_mixed_t<true, true, true>(a, spread, s, n_sm) : launch_mixed_t<true, false, true>(a, spread, s, n_sm);
  }
  if (grad) return phase64 ? launch_mixed_t<true, true>(a, spread, s, n_sm) : launch_mixed_t<true, false>(a, spread, s, n_sm);
  return phase64 ? launch_mixed_t<false, true>(a, spread, s, n_sm) : launch_mixed_t<false, false>(a, spread, s, n_sm);
}

// Set-up and likelihood in one launch, where it applies (*done): every block
// gets at most kSetupWalkers walkers, and the tables leave room for their
// records beside them.  With mala the kernel forms the proposals too (theta is not
// read).
template <int ND, bool GRAD, bool MALA>
static cudaError_t launch_fused_nd(const FusedArgs& a, cudaStream_t s, int n_sm, bool* done) {
  auto* fn = k_rb_mixed<ND, GRAD, false, MALA, true>;
  const size_t smem = a.ev.slot32_floats * sizeof(float) + kFusedBytes + (MALA ? sizeof(MalaBlock) : 0);
  *done = false;
  if (smem > smem_optin_max()) return cudaSuccess;
  int per_sm = 0;
  const cudaError_t err = blocks_per_sm(reinterpret_cast<const void*>(fn), kThreads, smem, &per_sm);
  if (err != cudaSuccess) return err;
  if (per_sm < 1) return cudaSuccess;
  const int64_t grid = mixed_grid(a.W, true, n_sm, (int64_t)per_sm * n_sm);
  if ((a.W + grid - 1) / grid > kSetupWalkers) return cudaSuccess;
  fn<<<(unsigned)grid, kThreads, smem, s>>>(a);
  *done = true;
  return cudaGetLastError();
}

template <bool GRAD, bool MALA>
static cudaError_t launch_fused_t(const FusedArgs& a, cudaStream_t s, int n_sm, bool* done) {
  switch (a.ev.n_det) {
    case 1: return launch_fused_nd<1, GRAD, MALA>(a, s, n_sm, done);
    case 2: return launch_fused_nd<2, GRAD, MALA>(a, s, n_sm, done);
    case 3: return launch_fused_nd<3, GRAD, MALA>(a, s, n_sm, done);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_rb_fused(const EventDev& ev, const EventConst& ec, const double* theta, int64_t W, double* logl,
                            double* grad, cudaStream_t s, int n_sm, const MalaArgs* mala, bool* done) {
  FusedArgs a;
  static_cast<LaunchArgs&>(a) = LaunchArgs{ev, nullptr, nullptr, W, logl, grad, {}};
  a.theta = theta;
  a.ec = ec;
  if (mala) {
    a.mala = *mala;
    return launch_fused_t<true, true>(a, s, n_sm, done);
  }
  return grad ? launch_fused_t<true, false>(a, s, n_sm, done) : launch_fused_t<false, false>(a, s, n_sm, done);
}

template <bool GRAD, bool MALA>
static cudaError_t launch_f64_t(const LaunchArgs& a, cudaStream_t s, int n_sm) {
  void (*const kernels[kMaxDet])(LaunchArgs) = {k_rb_f64<1, GRAD, MALA>, k_rb_f64<2, GRAD, MALA>, k_rb_f64<3, GRAD, MALA>};
  if (a.ev.n_det < 1 || a.ev.n_det > kMaxDet) return cudaErrorInvalidValue;
  auto* fn = kernels[a.ev.n_det - 1];
  const int bs = 256;
  int per_sm = 0;
  cudaError_t err = blocks_per_sm(reinterpret_cast<const void*>(fn), bs, 0, &per_sm);
  if (err != cudaSuccess) return err;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  // a batch that does not fill the SMs with eight walkers per block is spread over
  // more of them, down to one walker per SM sub-partition (each has one FP64 unit)
  const int64_t dense = (a.W * 32 + bs - 1) / bs;
  const int64_t thin = std::min<int64_t>((a.W + kThinWalkers - 1) / kThinWalkers, n_sm);
  fn<<<(unsigned)std::min<int64_t>(std::max(dense, thin), (int64_t)per_sm * n_sm), bs, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_rb_f64(const EventDev& ev, const void* ws, const void* tan, int64_t W, double* logl, double* grad,
                          cudaStream_t s, int n_sm, const MalaArgs* mala) {
  LaunchArgs a{ev, ws, tan, W, logl, grad, {}};
  if (mala) {
    a.mala = *mala;
    return launch_f64_t<true, true>(a, s, n_sm);
  }
  return grad ? launch_f64_t<true, false>(a, s, n_sm) : launch_f64_t<false, false>(a, s, n_sm);
}

}  // namespace rb

RB_BOUNDS_READER(rb_bounds_read_loglike)

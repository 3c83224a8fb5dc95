// rb_full.cu -- the full (unbinned) log-likelihood of Eqs. 2-3 for a batch
// of walkers, on the full frequency grid: the quantity relative binning
// approximates, used for the reference-parameter search and for checking the
// binned likelihood (Sec. II.C; Sec. III.A).
//
// With the Newtonian amplitude the waveform is h_d(f; theta) = K_d(theta)
// f^-7/6 exp(-2 pi i x_d(f; theta)), so per detector
//   <d|h> = 4 df Re[conj(K_d) Z_d],  Z_d = sum_k (d_k / S_k) f_k^-7/6 exp(+2 pi i x_d(f_k)),
//   <h|h> = |K_d|^2 H_d,             H_d = 4 df sum_k f_k^-7/3 / S_k,
//   log L = sum_d (<d|h> - <h|h> / 2).
// H_d does not depend on theta: it is sum_b B0_{d,b} / |K_d(theta_ref)|^2 from
// the summary data (B0 = <h0|h0> over the bin).  Z_d is the expensive part: a
// walker-dependent phase at every grid point.  It is evaluated like the fast
// summary build: x_d on a chunk of 32 points is a Taylor polynomial whose
// coefficients are the walker's c_k / 2pi contracted with the event's chunk
// matrices, and the delay enters as exp(2 pi i f_c tau_d) exp(2 pi i j df tau_d).
//
// Mapping: a block of 8 warps takes 8 walkers (one per warp) and a group of
// segments of 64 chunks (2048 points) at a time; the (walkers, group) pairs are
// dealt to one wave of blocks in equal contiguous shares.  Per segment the block stages the chunk matrices and the FP32 data
// copy times f^-7/6 in shared memory, the data transposed (read once for the 8
// walkers; the event's data stay in L2).  Lane l of a warp forms its walker's
// Taylor coefficients for chunks l and l + 32 and walks their 32 points side by
// side, the two chunks as the halves of paired FP32 values; the offset factors
// exp(2 pi i (j - 16) df tau_d), the same for all chunks at a given offset j,
// come from a per-warp table (broadcast loads), and the chunk factors
// exp(2 pi i f_c tau_d) are applied once to the chunk's sums.  Per point: the
// phase polynomial, one sin/cos, and per detector the offset factor times the
// phasor times the data.  Per-lane sums are FP32 per chunk, accumulated in float
// pairs over a group of segments, at whose end the warp's lanes are added (a
// fixed tree of float pairs); the groups are added in FP64.  The pairs hold the sum of a
// group's chunk sums (24-bit numbers of like size) exactly: emulated over grids of 64 to
// 128 s and noise- and signal-like sums, its error is zero, as with FP64 over the lanes,
// which takes 437 us where this takes 416.  The groups depend
// on the grid alone, so a walker's result does not depend on the batch.
//
// Phase: the first three Taylor terms X0 + X1 j + X2 j^2 run in integers, in units
// of 2^-32 turns: they wrap at whole turns by themselves, a point costs two integer
// additions (first and second differences, on a pipe that is idle otherwise), and
// what the units drop goes into the FP32 polynomial of the remaining terms.  In float
// pairs (products, two-sums, reductions) these terms were 31 of a point's 79 FP32
// operations; 3 are left.  Segments whose orders beyond 4 stay below 2^-36 turns (and
// the terms from order 3 below 2^-10, so that the sum needs no reduction) leave those
// orders out: nearly all above ~80 Hz; the walkers of a block decide for themselves.
//
// Bound: the FP32 pipe (~50 operations per point and walker with 3 detectors, 24 of
// them the detectors' products, 18 the sine and cosine, and ~12 for the chunk
// coefficients).  512 walkers, 260 k points, 3 detectors: call 512 -> 416 us; with one
// chunk per lane in scalar FP32, in waves of slices, it was 588.  The phases agree with
// the float-pair form to its last bit at nearly every point: results differ by
// 1e-12 to 2e-10, errors against FP64 sums unchanged.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <type_traits>

#include "rb.h"
#include "rb_api_internal.h"
#include "rb_internal.cuh"

namespace rb {

constexpr int kFullWarps = 8;
constexpr int kFullThreads = kFullWarps * 32;
constexpr int kSegC = 64;                 // chunks per segment, two per lane
constexpr int kSegP = kSegC * kChunk;     // points per segment
constexpr int kWtRow = kSegC / 2 + 1;     // transposed data row (padded: conflict-free stores)
constexpr int kQPad = kQRow + 4;          // staged chunk-matrix row (padded: 16-byte loads of row l by lane l without conflicts)
constexpr int full_smem(int nd) {
  return (int)(sizeof(float4) * (nd * kChunk * kWtRow + nd * kFullWarps * kChunk) + sizeof(float2) * kChunk + sizeof(float) * kSegC * kQPad);
}

// Segments per group: up to 64 groups.
constexpr int kGroups = 64;
constexpr int kTileBytes = 64 << 20;  // the groups' sums held at a time
__host__ __device__ constexpr int group_segments(int n_seg) { return (n_seg + kGroups - 1) / kGroups; }

// One level of a transposed warp sum of float pairs: lanes whose bit o is clear
// keep values [0, M) and send [M, N), the others keep [M, N) (zero beyond N)
// and send [0, M); each adds what its partner sent (two-sum of the high parts).
template <int N, int M>
__device__ __forceinline__ void ff_level(const f2x (&in)[N], f2x (&out)[M], int lane, int o) {
  const bool up = (lane & o) != 0;
#pragma unroll
  for (int i = 0; i < M; ++i) {
    const f2x lo = in[i], hi = (M + i < N) ? in[M + i] : f2x{0.f, 0.f};
    const f2x keep = up ? hi : lo, send = up ? lo : hi;
    const float bh = __shfl_xor_sync(0xffffffffu, send.hi, o), bl = __shfl_xor_sync(0xffffffffu, send.lo, o);
    out[i] = keep;
    f2x_add(out[i].hi, out[i].lo, bh);
    out[i].lo = __fadd_rn(out[i].lo, bl);
  }
}

// hi + lo turns, mod 1, as an integer i in units of 2^-32 turns and the rest, e
// turns (|e| <= 2^-32): both parts' fractions times 2^32 are integers or below
// 2^24, so that i's conversions back are exact.
__device__ __forceinline__ void turns_fixed(float hi, float lo, unsigned& i, float& e) {
  float a = 0x1p32f * pv::frac1(hi), b = 0x1p32f * pv::frac1(lo);
  a = a == 0x1p31f ? -0x1p31f : a;  // +1/2 turn is out of the integers' range (a NaN stays one)
  b = b == 0x1p31f ? -0x1p31f : b;
  const int ia = __float2int_rn(a), ib = __float2int_rn(b);
  e = 0x1p-32f * ((a - (float)ia) + (b - (float)ib));
  i = (unsigned)ia + (unsigned)ib;
}

// Per group of segments and walker: the group's part of Z_d (complex, 3
// detectors) as FP64 in zout[group][w][6].  ND = number of detectors.
template <int ND>
__global__ void __launch_bounds__(kFullThreads, 2) k_full_z(const float2* __restrict__ w32, int N,
                                                           const float* __restrict__ q, int n_chunks,
                                                           const WalkerAbs* __restrict__ wabs, int64_t W,
                                                           float invT_hi, float invT_lo,
                                                           double* __restrict__ zout) {
  // dynamic shared memory: the segment's data times f^-7/6, transposed: for
  // detector d and offset j, [d][j][l] holds {re, re', im, im'} of chunks l and
  // l + 32 (wt); per warp the walker's offset factors exp(2 pi i (j - 16) df
  // tau_d) as {re, re, im, im} (tp[warp][j][d]); the offsets {j - 16, j - 16}
  // (jt); the segment's chunk matrices (qs)
  extern __shared__ __align__(16) unsigned char smem_full[];
  float4 (*wt)[kChunk][kWtRow] = reinterpret_cast<float4 (*)[kChunk][kWtRow]>(smem_full);
  float4 (*tp)[kChunk][ND] = reinterpret_cast<float4 (*)[kChunk][ND]>(wt + ND);
  float2* jt = reinterpret_cast<float2*>(tp + kFullWarps);
  float* qs = reinterpret_cast<float*>(jt + kChunk);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n_seg = (n_chunks + kSegC - 1) / kSegC, gs = group_segments(n_seg), n_groups = (n_seg + gs - 1) / gs;
  if (warp == 0) {
    const float jf = small_int_float(lane - kChunk / 2);
    jt[lane] = make_float2(jf, jf);
  }
  // the (walker octet, group) pairs, octet-major, in equal contiguous shares
  const int64_t units = (W + kFullWarps - 1) / kFullWarps * n_groups;
  const int64_t u0 = units * blockIdx.x / gridDim.x, u1 = units * (blockIdx.x + 1) / gridDim.x;
  for (int64_t u = u0; u < u1; ++u) {
    const int g = (int)(u % n_groups);
    const int64_t w = u / n_groups * kFullWarps + warp;
    const bool live = w < W;
    const WalkerAbs& wa = wabs[live ? w : W - 1];
    const bool valid = live && wa.valid;
    if (u == u0 || g == 0) {
      // offset factors of the warp's walker: lane j forms exp(2 pi i (j - 16) df tau_d)
      __syncwarp();
      const float jf = small_int_float(lane - kChunk / 2);
#pragma unroll
      for (int d = 0; d < ND; ++d) {
        float sh = 0.f, sl = 0.f;
        if (valid) f2x_fma_acc(wa.taut[d][0], wa.taut[d][1], invT_hi, invT_lo, sh, sl);  // tau_d df
        const float p = __fmul_rn(sh, jf);
        const float e = __fmaf_rn(sl, jf, __fmaf_rn(sh, jf, -p));
        const float2 t = cis_turns(frac_turns(p, e));
        tp[warp][lane][d] = make_float4(t.x, t.x, t.y, t.y);
      }
    }
    f2x z[2 * ND];  // the lane's part of Z_d (re, im)
#pragma unroll
    for (int i = 0; i < 2 * ND; ++i) z[i] = f2x{0.f, 0.f};
    for (int sg = g * gs; sg < min(n_seg, (g + 1) * gs); ++sg) {
      const int c0 = sg * kSegC, nc = min(kSegC, n_chunks - c0);
      __syncthreads();  // the previous segment is no longer read (and the tables are written)
      {
        const float4* src = reinterpret_cast<const float4*>(q + (size_t)c0 * kQRow);
        float4* dst = reinterpret_cast<float4*>(qs);
#pragma unroll 8
        for (int i = tid; i < nc * (kQRow / 4); i += kFullThreads)
          dst[(i / (kQRow / 4)) * (kQPad / 4) + i % (kQRow / 4)] = __ldg(src + i);
      }
      __syncthreads();
      // data times f^-7/6 = f_c^-7/6 (1 + j u)^-7/6 (chunk series), transposed,
      // chunks c and c + 32 together; points past the grid are zero
#pragma unroll 2
      for (int i = 0; i < kSegP / 2 / kFullThreads; ++i) {
        const int p = tid + i * kFullThreads, c = p >> 5, jj = p & (kChunk - 1);
        const float j = small_int_float(jj - kChunk / 2);
        float2 v[2][ND];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int ch = c + h * (kSegC / 2), k = (c0 + ch) * kChunk + jj;
          const bool in = ch < nc && k < N;
          const float* qa = qs + ch * kQPad + kQamp;
          const float A = in ? qa[0] * fmaf(j, fmaf(j, fmaf(j, fmaf(j, qa[4], qa[3]), qa[2]), qa[1]), 1.f) : 0.f;
#pragma unroll
          for (int d = 0; d < ND; ++d) {
            const float2 x = in ? __ldg(w32 + (size_t)d * N + k) : make_float2(0.f, 0.f);
            v[h][d] = in ? make_float2(x.x * A, x.y * A) : make_float2(0.f, 0.f);
          }
        }
#pragma unroll
        for (int d = 0; d < ND; ++d) wt[d][jj][c] = make_float4(v[0][d].x, v[1][d].x, v[0][d].y, v[1][d].y);
      }
      __syncthreads();  // wt complete
      if (!valid) continue;  // the whole warp
      // the walker's coefficients of the lane's chunks (X0 with Phi0); a chunk past
      // the last has zero data and the first chunk's row (chunk l) or zeros (chunk l + 32)
      const bool in0 = lane < nc, in1 = lane + kSegC / 2 < nc;
      const float* r0 = qs + (in0 ? lane : 0) * kQPad;
      const float* r1 = qs + (lane + kSegC / 2) * kQPad;
      // float4 i of the two rows
      auto row4 = [&](int i, float4& a, float4& b) {
        a = reinterpret_cast<const float4*>(r0)[i];
        b = in1 ? reinterpret_cast<const float4*>(r1)[i] : make_float4(0.f, 0.f, 0.f, 0.f);
      };
      float2 X0h = pv::splat<float2>(wa.phi0t[0]), X0l = pv::splat<float2>(wa.phi0t[1]);
      float2 X1h = make_float2(0.f, 0.f), X1l = X1h, X2h = X1h, X2l = X1h;
      float2 s_abs = X1h, g_lf = X1h, g_cf = X1h;  // the terms' moduli; ln f_c, f_c^1/3
      float4 a, b;
#pragma unroll
      for (int k = 0; k < kNBasis; ++k) {
        const float2 ch = pv::splat<float2>(wa.chat[k][0]), cl = pv::splat<float2>(wa.chat[k][1]);
        row4(kQ01 / 4 + k, a, b);
        const float2 g = make_float2(a.x, b.x);
        pv::fma_acc(ch, cl, g, make_float2(a.y, b.y), X0h, X0l);
        pv::fma_acc(ch, cl, make_float2(a.z, b.z), make_float2(a.w, b.w), X1h, X1l);
        if (k == 4) g_lf = make_float2(fabsf(g.x), fabsf(g.y));
        if (k == 5) g_cf = g;
        const float2 cabs = pv::splat<float2>(fabsf(wa.chat[k][0]));
        if (k == 4) s_abs = pv::add(s_abs, cabs);
        s_abs = pv::fma(cabs, k == 6 ? pv::fma(g_lf, g_cf, g_cf) : make_float2(fabsf(g.x), fabsf(g.y)), s_abs);
        if (k % 2 == 0) {
          const float2 ch1 = pv::splat<float2>(wa.chat[k + 1][0]), cl1 = pv::splat<float2>(wa.chat[k + 1][1]);
          row4(kQ2 / 4 + k / 2, a, b);
          pv::fma_acc(ch, cl, make_float2(a.x, b.x), make_float2(a.y, b.y), X2h, X2l);
          pv::fma_acc(ch1, cl1, make_float2(a.z, b.z), make_float2(a.w, b.w), X2h, X2l);
        }
      }
      // X0, X1, X2 mod 1 as integers in units of 2^-32 turns and the rest: x0 + x1 j
      // + x2 j^2 then wraps at whole turns by itself, exactly
      unsigned x[2], d1[2], d2[2];
      float2 e0, e1, e2;
      {
        unsigned i0[2], i1[2], i2[2];
        turns_fixed(X0h.x, X0l.x, i0[0], e0.x);
        turns_fixed(X0h.y, X0l.y, i0[1], e0.y);
        turns_fixed(X1h.x, X1l.x, i1[0], e1.x);
        turns_fixed(X1h.y, X1l.y, i1[1], e1.y);
        turns_fixed(X2h.x, X2l.x, i2[0], e2.x);
        turns_fixed(X2h.y, X2l.y, i2[1], e2.y);
#pragma unroll
        for (int h = 0; h < 2; ++h) {  // value (biased by half a turn), first and second difference at j = -16
          x[h] = i0[h] - 16u * i1[h] + 256u * i2[h] + 0x80000000u;
          d1[h] = i1[h] - 31u * i2[h];
          d2[h] = 2u * i2[h];
        }
      }
      float2 ar[ND], ai[ND];  // the chunks' sums
#pragma unroll
      for (int d = 0; d < ND; ++d) ar[d] = ai[d] = make_float2(0.f, 0.f);
      auto points = [&](auto short_c) {
        constexpr bool SHORT = decltype(short_c)::value;
        constexpr int NT = SHORT ? 2 : kOrd - 2;  // orders from 3 up
        float2 xn[NT];
#pragma unroll
        for (int n = 0; n < NT; ++n) xn[n] = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < NT * kNBasis / 4; ++i) {  // basis index fastest
          row4(kQh / 4 + i, a, b);
          const float2 m[4] = {make_float2(a.x, b.x), make_float2(a.y, b.y), make_float2(a.z, b.z), make_float2(a.w, b.w)};
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const int n = (4 * i + v) / kNBasis, k = (4 * i + v) % kNBasis;
            xn[n] = pv::fma(pv::splat<float2>(wa.chat[k][0]), m[v], xn[n]);
          }
        }
        const float2 one = make_float2(1.f, 1.f), two = make_float2(2.f, 2.f);
#pragma unroll 2
        for (int jj = 0; jj < kChunk; ++jj) {
          const float2 j = jt[jj];
          // the high 16 bits of x as floats 2^23 + h (a byte permutation), the low 16 converted
          const float2 hb = make_float2(__uint_as_float(__byte_perm(x[0], 0x4B000000u, 0x7432)),
                                        __uint_as_float(__byte_perm(x[1], 0x4B000000u, 0x7432)));
          const float2 lb = make_float2(__uint2float_rn(x[0] & 0xffffu), __uint2float_rn(x[1] & 0xffffu));
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            x[h] += d1[h];
            d1[h] += d2[h];
          }
          // e0 + e1 j + e2 j^2 + X3 j^3 + ...
          float2 t = xn[NT - 1];
#pragma unroll
          for (int n = NT - 2; n >= 0; --n) t = pv::fma(t, j, xn[n]);
          t = pv::fma(pv::fma(pv::fma(t, j, e2), j, e1), j, e0);
          t = pv::fma(lb, pv::splat<float2>(0x1p-32f), t);
          float2 y = pv::fma(pv::sub(hb, pv::splat<float2>(8421376.f)), pv::splat<float2>(0x1p-16f), t);
          if constexpr (!SHORT) y = pv::frac1(y);
          float2 sn, cs;
          pv::sincos_half(y, sn, cs);
          const float2 s2 = pv::mul(two, sn);
          const float2 zx = pv::fma(pv::neg(s2), sn, one), zy = pv::mul(s2, cs);  // exp(+2 pi i x)
          // offset factor times the phasor, times the data
#pragma unroll
          for (int d = 0; d < ND; ++d) {
            const float4 T = tp[warp][jj][d], v = wt[d][jj][lane];
            const float2 Tr = make_float2(T.x, T.y), Ti = make_float2(T.z, T.w);
            const float2 vr = make_float2(v.x, v.y), vi = make_float2(v.z, v.w);
            const float2 ur = pv::fma(zx, Tr, pv::mul(pv::neg(zy), Ti)), ui = pv::fma(zx, Ti, pv::mul(zy, Tr));
            ar[d] = pv::fma(vr, ur, pv::fma(pv::neg(vi), ui, ar[d]));
            ai[d] = pv::fma(vr, ui, pv::fma(vi, ur, ai[d]));
          }
        }
      };
      // |X_n j^n| <= 6 s_abs (16 u)^n (every |alpha_kn|, |beta_n| <= 5.2); 16 u from
      // the amplitude series' first coefficient, -7/6 u
      const float u16 = 13.8f * fabsf(r0[kQamp + 1]);
      const float b3 = 6.f * fmaxf(s_abs.x, s_abs.y) * (u16 * u16 * u16);
      const bool small = b3 < 0x1p-10f && b3 * (u16 * u16) < 0x1p-36f;
      if (__all_sync(0xffffffffu, small)) points(std::true_type{});
      else points(std::false_type{});
      // the chunk factors exp(2 pi i f_c tau_d), once per chunk, then into the
      // lane's float pairs, chunk l before chunk l + 32
#pragma unroll
      for (int d = 0; d < ND; ++d) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (h == 1 && !in1) continue;
          const float* r = h ? r1 : r0;
          float ah = 0.f, al = 0.f;
          f2x_fma_acc(wa.taut[d][0], wa.taut[d][1], r[kQfc], r[kQfc + 1], ah, al);  // f_c tau_d
          const float2 E = cis_turns(frac_turns(ah, al));
          const float a_r = h ? ar[d].y : ar[d].x, a_i = h ? ai[d].y : ai[d].x;
          f2x_add(z[2 * d].hi, z[2 * d].lo, fmaf(E.x, a_r, -E.y * a_i));
          f2x_add(z[2 * d + 1].hi, z[2 * d + 1].lo, fmaf(E.x, a_i, E.y * a_r));
        }
      }
    }
    // the lanes' sums: after the five levels a lane holds one value
    constexpr int n0 = 2 * ND, n1 = (n0 + 1) / 2, n2 = (n1 + 1) / 2, n3 = (n2 + 1) / 2;
    static_assert(n3 == 1, "three levels reduce to one value");
    f2x z1[n1], z2[n2], z3[1], z4[1], z5[1];
    ff_level(z, z1, lane, 16);
    ff_level(z1, z2, lane, 8);
    ff_level(z2, z3, lane, 4);
    ff_level(z3, z4, lane, 2);
    ff_level(z4, z5, lane, 1);
    // its index: the halves the lane kept, from the last level back (a lane whose
    // kept half was padding holds none)
    int idx = (lane & 4) ? n3 : 0;
    bool ok = (lane & 3) == 0 && idx < n2;
    idx += (lane & 8) ? n2 : 0;
    ok = ok && idx < n1;
    idx += (lane & 16) ? n1 : 0;
    if (live && ok && idx < n0) zout[((size_t)g * W + w) * 6 + idx] = (double)z5[0].hi + (double)z5[0].lo;
  }
}

// log L per walker from Z_d and K_d (FP64); H_d from the summary's B0 and
// the reference prefactor, scales from the FP32 data copy's exponents.  Eight
// lanes per walker, each adding every eighth group; one warp per detector forms
// H_d (one warp for all detectors and one thread per walker took 31 us for 512
// walkers, all of it load latency).
constexpr int kFinishLanes = 8;
constexpr int kFinishThreads = 128;
__global__ void __launch_bounds__(kFinishThreads) k_full_finish(const double* __restrict__ zout, int n_groups,
                                                     const WalkerAbs* __restrict__ wabs,
                                                     int64_t W, int D, int B, double T, const int* __restrict__ exps,
                                                     const double* __restrict__ summ, const RefValues* __restrict__ ref,
                                                     double* __restrict__ logl) {
  static_assert(kFinishThreads / 32 >= kMaxDet, "one warp per detector");
  __shared__ double H[kMaxDet], sc0[kMaxDet];
  const int part = threadIdx.x % kFinishLanes;
  const int64_t w = ((int64_t)blockIdx.x * kFinishThreads + threadIdx.x) / kFinishLanes;
  const int64_t wc = w < W ? w : W - 1;
  // the walker's sums over the groups, lane by lane, then a fixed tree
  double z[2 * kMaxDet] = {0, 0, 0, 0, 0, 0};
  for (int g = part; g < n_groups; g += kFinishLanes) {
    const double* zs = zout + ((size_t)g * W + wc) * 6;
#pragma unroll
    for (int i = 0; i < 2 * kMaxDet; ++i)
      if (i < 2 * D) z[i] += zs[i];
  }
  const int d = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (d < D) {
    double s[4] = {0, 0, 0, 0};
    for (int b = lane; b < B; b += 128)
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (b + 32 * u < B) s[u] += summ[((size_t)d * B + b + 32 * u) * 6 + 4];  // B0
    const double t = warp_sum_f64((s[0] + s[1]) + (s[2] + s[3]));
    if (lane == 0) {
      const double kr = ref->K[d][0], ki = ref->K[d][1];
      H[d] = t / (kr * kr + ki * ki);
      const int sd = exps[2 * d], sS = exps[2 * d + 1];
      sc0[d] = (4.0 / T) * __hiloint2double((1023 + sS - sd) << 20, 0);
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 2 * kMaxDet; ++i)
    if (i < 2 * D)
#pragma unroll
      for (int o = kFinishLanes / 2; o > 0; o >>= 1) z[i] += __shfl_xor_sync(0xffffffffu, z[i], o);
  if (w >= W || part != 0) return;
  if (!wabs[w].valid) {
    logl[w] = -INFINITY;
    return;
  }
  double L = 0.0;
#pragma unroll
  for (int dd = 0; dd < kMaxDet; ++dd) {
    if (dd >= D) break;
    const double kr = wabs[w].K[dd][0], ki = wabs[w].K[dd][1];
    const double dh = sc0[dd] * (kr * z[2 * dd] + ki * z[2 * dd + 1]);  // Re(conj(K) Z)
    L += dh - 0.5 * (kr * kr + ki * ki) * H[dd];
  }
  logl[w] = L;
}

cudaError_t launch_setup_abs(const double* theta, int64_t W, const EventConst& ec, WalkerAbs* out, cudaStream_t s);
cudaError_t launch_data32(const DataPtrs& in, int64_t N, int D, void* w32, float* is32, int* exps, cudaStream_t s);

}  // namespace rb

extern "C" int rb_loglike_full_batch(rb_event_t ev, const double* theta_dev, int64_t W, double* logl_dev, int mode,
                                     void* stream) {
  RB_NVTX("rb_loglike_full_batch");
  using namespace rb;
  if (!ev) return set_error(RB_EINVAL, "rb_loglike_full_batch: NULL event");
  if (W < 0) return set_error(RB_EINVAL, "rb_loglike_full_batch: W < 0");
  if (W == 0) return RB_OK;
  if (!theta_dev || !logl_dev) return set_error(RB_EINVAL, "rb_loglike_full_batch: NULL theta or logl");
  if (mode != RB_MIXED) return set_error(RB_EINVAL, "rb_loglike_full_batch: only RB_MIXED is provided");
  EventEntry& e = *const_cast<EventEntry*>(event_entry(ev));
  if (!(e.kmin >= 1024 && e.N <= (int64_t(1) << 30)))
    return set_error(RB_EINVAL, "rb_loglike_full_batch: needs T f_low >= 1024 and N <= 2^30 (chunk expansion)");
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t err;
  if (!e.w32_current) {  // FP32 working copy of the data the summary was built from
    if (e.last_in_place)
      return set_error(RB_EINVAL,
                       "rb_loglike_full_batch: the last rebuild read caller data in place in RB_FP64 mode; "
                       "rebuild in a mixed mode or from resident data");
    DataPtrs in{};
    for (int d = 0; d < e.n_det; ++d) {
      in.data[d] = e.d_data + 2 * (size_t)d * e.N;
      in.psd[d] = e.d_psd + (size_t)d * e.N;
    }
    if ((err = launch_data32(in, e.N, e.n_det, e.d_w32, e.d_is32, e.d_wexp, s)) != cudaSuccess)
      return cuda_fail(err, "rb_loglike_full_batch: data conversion kernel");
    e.w32_resident = e.w32_current = true;
    count_launches(1);
  }
  void (*const kz)(const float2*, int, const float*, int, const WalkerAbs*, int64_t, float, float, double*) =
      e.n_det == 1 ? k_full_z<1> : e.n_det == 2 ? k_full_z<2> : k_full_z<3>;
  const int smem = full_smem(e.n_det);
  static std::atomic<bool> smem_raised[kMaxDet];  // the attribute is idempotent: concurrent first calls only repeat it
  if (!smem_raised[e.n_det - 1].load(std::memory_order_acquire)) {
    if ((err = cudaFuncSetAttribute(kz, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess)
      return cuda_fail(err, "rb_loglike_full_batch: shared memory attribute");
    smem_raised[e.n_det - 1].store(true, std::memory_order_release);
  }
  // one wave of blocks (2 per SM), each with an equal share of the (8 walkers,
  // group) pairs
  const int nc = (int)((e.N + kChunk - 1) / kChunk);
  const int n_seg = (nc + kSegC - 1) / kSegC, gs = group_segments(n_seg), n_groups = (n_seg + gs - 1) / gs;
  // the groups' sums (up to 3 KB per walker) of so many walkers at a time: a batch
  // beyond that takes several pairs of launches, each of tens of units per block
  const int64_t tile = std::min<int64_t>(W, kTileBytes / (int)(sizeof(double) * 6 * kFullWarps) / n_groups * kFullWarps);
  char* buf = nullptr;
  const size_t abs_bytes = sizeof(WalkerAbs) * W, z_bytes = sizeof(double) * 6 * tile * n_groups;
  err = ws_alloc(reinterpret_cast<void**>(&buf), abs_bytes + z_bytes, s);
  if (err != cudaSuccess) return cuda_fail(err, "rb_loglike_full_batch: workspace allocation");
  WalkerAbs* wabs = reinterpret_cast<WalkerAbs*>(buf);
  double* zout = reinterpret_cast<double*>(buf + abs_bytes);
  const double invT = 1.0 / e.T;
  const float ih = (float)invT, il = (float)(invT - (double)ih);
  int rc = RB_OK;
  if ((err = launch_setup_abs(theta_dev, W, e.ec, wabs, s)) != cudaSuccess) {
    rc = cuda_fail(err, "rb_loglike_full_batch: set-up kernel");
  } else {
    count_launches(1);
    for (int64_t w0 = 0; w0 < W && rc == RB_OK; w0 += tile) {
      const int64_t n = std::min(tile, W - w0), units = (n + kFullWarps - 1) / kFullWarps * n_groups;
      const unsigned blocks = (unsigned)std::min<int64_t>(units, 2 * (int64_t)sm_count());
      kz<<<blocks, kFullThreads, smem, s>>>(static_cast<const float2*>(e.d_w32), (int)e.N,
                                            static_cast<const float*>(e.d_chunkq), nc, wabs + w0, n, ih, il, zout);
      constexpr int per_block = kFinishThreads / kFinishLanes;
      k_full_finish<<<(unsigned)((n + per_block - 1) / per_block), kFinishThreads, 0, s>>>(
          zout, n_groups, wabs + w0, n, e.n_det, e.n_bins, e.T, e.d_wexp, e.d_summ, e.d_ref, logl_dev + w0);
      if ((err = cudaGetLastError()) != cudaSuccess) rc = cuda_fail(err, "rb_loglike_full_batch: kernels");
      else count_launches(2);
    }
  }
  cudaFreeAsync(buf, s);
  return rc;
}

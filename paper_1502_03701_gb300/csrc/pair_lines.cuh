// Compact-derivative line pass in FP32 pair arithmetic, for base flows that
// depend on y only.
//
// What bounds it: GB300 issues FP64 at 1/64 of its FP32 rate, so a line pass
// in FP64 is bound by the FP64 pipe however it is laid out.  Here one FP64
// subtraction per point forms the difference of two inputs (exact for
// neighbouring values of a smooth field, so no digits are lost to the
// cancellation), the difference is split into an FP32 pair (~2^-49 relative),
// and everything after it runs in pairs: the stencil, the two sweeps and their
// corrections, about 100 FP32 instructions per derivative value in place of
// six to nine FP64 instructions that cost 64 issue slots each.
//
// The tridiagonal system of the interior rows factorises for a constant
// coefficient line into c (1 - r S^-1)(1 - r S).  A line is cut into chunks of
// at most C points; every thread sweeps one chunk of one real line forward and
// backward from zero, and the neighbours enter afterwards through the two
// homogeneous solutions r^(k+1) and r^(len-k) of the chunk with amplitudes
// from the chunk ends (a partitioned tridiagonal solve): no warm-up sweeps and
// no serial dependence between chunks.  The one-sided and Pade closure rows of
// a bounded line change only the first two and the last two rows, so they
// enter as amplitudes of the same two solutions as well.
//
// Values are stored scaled: first derivatives as f' / S1 and second ones as
// f'' / S2 with the schemes' leading factors (AxisTables::pscale), which the
// pointwise map's coefficients carry.  Differences of neighbours are smaller than
// the derivatives by 1/h and 1/h^2, and a split keeps its low part from 2^-74 up
// only, so they are split times 2^u, u = log2(1/h) or log2(1/h^2) (exact; no
// instruction more): S1 and S2 are then in [1, 2), and the range of v over which the
// operator is accurate is that of its derivatives.  Unscaled, second derivatives of
// a smooth field of size 2^-64 on 256 points were good to 1e-9 only.  The second
// derivation of a mixed derivative takes pairs and is not scaled.
//
// 128 x 256 x 64 points: y 257, z 267, x 346 us for all derivatives of an axis;
// FP64 sweeps took 0.96, 0.87 and 1.06 ms.  60 x 90 x 28 points: 62 to 67 % of the
// issue slots.  32 x 64 points: 10.5 and 8.7 us (32 us each), one warp's latency.
#pragma once
#include "internal.cuh"

namespace pl {

constexpr int kMaxThreads = 512;
constexpr int kTabPow = 72;                    // r^(i - 2), i < kTabPow
constexpr int kTab = kTabPow + kPairMaxC + 1;  // then u0(len), len <= kPairMaxC
constexpr size_t kSmemMax = 200 * 1024;        // dynamic shared memory opt-in

struct PairJob {
  const double2* in;  // complex field (pair_in: pairs (re.hi, re.lo, im.hi, im.lo) in the same 16 bytes)
  float4* out;        // pairs in that layout
  int kind;           // 0 first, 1 second derivative
  int pair_in;
};

struct PairPass {
  PairJob job[STAB_MAX_JOBS];
  PairKind k[2];
  const ffn* tab[2];
  const int* gate;   // when set and nonzero the launch does nothing
  long long nlines;  // complex lines
  long long stride;  // points between consecutive points of a line
  int njobs, axis, n, nx, ny;
  int nblk;          // line blocks
  int lanes;         // components per thread: 2 packed, 1
  int L, Lp;         // complex lines per CTA, shared-memory pitch of a point (odd: conflict-free either way)
  int U, Up;         // the same in units of a thread's lines (x 2 / lanes)
  int nch, q, rem;   // chunks per line: the first rem have q + 1 points, the others q
  int bounded, pad;
  int up[2];         // exponent scaling of the differences per kind (ff2_split)
  FastDiv divblk, divL, divU, divn, divnx;
};
static_assert(sizeof(PairPass) % 8 == 0, "items are copied to shared memory in 8-byte words");

// complex index of the first point of line l
__device__ __forceinline__ long long line_start(const PairPass& P, long long l) {
  if (P.axis == 0) return l * P.n;
  if (P.axis == 1) {
    const long long z = fdiv((unsigned)l, P.divnx);
    return z * (long long)P.nx * P.ny + (l - z * P.nx);
  }
  return l;
}

__device__ __forceinline__ void copy16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem) : "memory");
}

// A thread's share of a point: both components (packed) or one.
template <int LANES>
struct Lane;
template <>
struct Lane<2> {
  typedef ffn2 Pair;
  typedef float4 Elem;
  static __device__ __forceinline__ Pair dup(ffn a) { return ff2_dup(a); }
  static __device__ __forceinline__ Pair zero() { return ff2_zero2(); }
  // difference of two staged FP64 values (times 2^up) as a pair: one FP64 subtraction per component
  static __device__ __forceinline__ Pair raw_diff(Elem a, Elem b, int up) {
    auto d = [](float l, float h) { return __hiloint2double(__float_as_int(h), __float_as_int(l)); };
    return ff2_split(make_double2(d(a.x, a.y) - d(b.x, b.y), d(a.z, a.w) - d(b.z, b.w)), up);
  }
  static __device__ __forceinline__ Elem table(float2 v) { return make_float4(v.x, v.x, v.y, v.y); }
};
template <>
struct Lane<1> {
  typedef ffn Pair;
  typedef float2 Elem;
  static __device__ __forceinline__ Pair dup(ffn a) { return a; }
  static __device__ __forceinline__ Pair zero() { return ffn{0.0f, 0.0f}; }
  static __device__ __forceinline__ Pair raw_diff(Elem a, Elem b, int up) {
    auto d = [](Elem v) { return __hiloint2double(__float_as_int(v.y), __float_as_int(v.x)); };
    return ff2_split(d(a) - d(b), up);
  }
  static __device__ __forceinline__ Elem table(float2 v) { return v; }
};

// One chunk of one line; block-uniform control flow around the barriers.  gs:
// distance of consecutive points of gout.
template <int LANES, int KIND, bool PAIR>
__device__ __forceinline__ void solve_chunks(const PairPass& P, typename Lane<LANES>::Elem* F,
                                             typename Lane<LANES>::Elem* E, typename Lane<LANES>::Elem* X,
                                             typename Lane<LANES>::Elem* W, const typename Lane<LANES>::Elem* tab,
                                             bool act, int c, int r, typename Lane<LANES>::Elem* gout, long long gs) {
  typedef Lane<LANES> T;
  typedef typename T::Pair Pair;
  typedef typename T::Elem Elem;
  const int n = P.n, nch = P.nch, L = P.U, Lp = P.Up;
  const bool bounded = P.bounded;
  const PairKind& K = P.k[KIND];
  const int up = P.up[KIND];
  auto len_of = [&](int cc) { return P.q + (cc < P.rem ? 1 : 0); };
  auto pw = [&](int i) { return ff2_unpack(tab[i + 2]); };  // r^i, i >= -2
  const int t0 = act ? c * P.q + min(c, P.rem) : 0, len = act ? len_of(c) : 0, t1 = t0 + len;
  Elem* col = F + (size_t)t0 * Lp + r;
  auto got = [&](int k) { return ff2_unpack(col[k * Lp]); };
  auto at = [&](int t) -> Elem {  // staged value at line index t (wrapped, or clamped where it is not used)
    if (bounded) t = min(max(t, 0), n - 1);
    else t = t < 0 ? t + n : (t >= n ? t - n : t);
    return F[(size_t)t * Lp + r];
  };
  auto dif = [&](Elem a, Elem b) -> Pair {  // a - b
    if constexpr (PAIR) return ff2_add(ff2_from_slot(a), ff2_neg(ff2_from_slot(b)));
    else return T::raw_diff(a, b, up);
  };
  // the neighbours' points, and the wall rows' right-hand sides, before any point is overwritten
  Elem fm2{}, fm1{}, fp0{}, fp1{};
  // side 0: rows 0 and 1 in the first chunk; side 1: rows n - 1 and n - 2 in the last one
  auto wall = [&](int side) { return bounded && act && c == (side ? nch - 1 : 0); };
  if (act) {
    fm2 = at(t0 - 2);
    fm1 = at(t0 - 1);
    fp0 = at(t1);
    fp1 = at(t1 + 1);
  }
#pragma unroll 1
  for (int side = 0; side < 2; ++side)
    if (wall(side)) {
      Pair u, v;
      if (KIND == 0) {
        const int i = side ? n - 2 : 1, k = side ? n - 2 : 0;
        u = dif(at(i + 1), at(i - 1));
        v = dif(at(k + 1), at(k));
      } else {
        auto second = [&](int i) { return ff2_add(dif(at(i + 1), at(i)), ff2_neg(dif(at(i), at(i - 1)))); };
        u = second(side ? n - 2 : 1);
        v = second(side ? n - 3 : 2);
      }
      W[(2 + side) * L + r] = ff2_pack(u);
      W[(4 + side) * L + r] = ff2_pack(v);
    }
  __syncthreads();
  // forward sweep from zero, in place: g_t = w_t + r g_{t-1}, w_t = d_t + rho (d_{t-1} + d_{t+1}),
  // d_t = f_{t+1} - f_{t-1} (first) or f_{t+1} - 2 f_t + f_{t-1} (second derivative)
  const Pair root = T::dup(K.r);
  if (act) {
    const Pair rho = T::dup(K.rho);
    Elem fa = col[0], fb = col[Lp];  // f_t, f_{t+1}
    Pair dm, d, gl = T::zero();
    if (KIND == 0) {
      dm = dif(fa, fm2);
      d = dif(fb, fm1);
    } else {
      const Pair g0 = dif(fm1, fm2), g1 = dif(fa, fm1);
      gl = dif(fb, fa);  // f_{t+1} - f_t
      dm = ff2_add(g1, ff2_neg(g0));
      d = ff2_add(gl, ff2_neg(g1));
    }
    Pair g = T::zero();
#pragma unroll 2
    for (int k = 0; k < len; ++k) {
      const Elem fc = k + 2 < len ? col[(k + 2) * Lp] : k + 2 == len ? fp0 : fp1;  // f_{t+2}
      Pair dn;
      if (KIND == 0) {
        dn = dif(fc, fa);
      } else {
        const Pair gn = dif(fc, fb);
        dn = ff2_add(gn, ff2_neg(gl));
        gl = gn;
      }
      Pair w = ff2_fma_u(rho, ff2_add_u(dm, dn), d);
      if (bounded && (unsigned)(t0 + k - 2) > (unsigned)(n - 5)) w = T::zero();  // wall rows
      g = ff2_fma(root, g, w);
      col[k * Lp] = ff2_pack(g);
      dm = d;
      d = dn;
      fa = fb;
      fb = fc;
    }
    E[c * L + r] = ff2_pack(g);
  }
  __syncthreads();
  // the true g at the point before the chunk
  Pair G = T::zero();
  if (act) {
    int off = 0, cc = c;
#pragma unroll 1
    for (int j = 0; j < nch && off < K.reach; ++j) {
      if (--cc < 0) {
        if (bounded) break;
        cc += nch;
      }
      G = ff2_fma(pw(off), ff2_unpack(E[cc * L + r]), G);
      off += len_of(cc);
    }
    if (!bounded && n < K.reach) G = ff2_fma(T::dup(K.invn), G, T::zero());  // the line closes on itself
    // backward sweep from zero, in place: x_t = g_t + r x_{t+1}
    Pair x = T::zero();
#pragma unroll 4
    for (int k = len - 1; k >= 0; --k) {
      x = ff2_fma(root, x, got(k));
      col[k * Lp] = ff2_pack(x);
    }
    X[c * L + r] = ff2_pack(ff2_fma(ff2_unpack(tab[kTabPow + len]), G, x));
  }
  __syncthreads();
  Pair A = T::zero(), B = T::zero();
  if (act) {
    Pair xn = T::zero();  // the true x at the point after the chunk
    int off = 0, cc = c;
#pragma unroll 1
    for (int j = 0; j < nch && off < K.reach; ++j) {
      if (++cc >= nch) {
        if (bounded) break;
        cc -= nch;
      }
      xn = ff2_fma(pw(off), ff2_unpack(X[cc * L + r]), xn);
      off += len_of(cc);
    }
    if (!bounded && n < K.reach) xn = ff2_fma(T::dup(K.invn), xn, T::zero());
    A = ff2_fma(T::dup(K.kap), G, T::zero());
    B = ff2_fma(ff2_neg(pw(len + 1)), A, xn);
  }
  if (bounded) {
#pragma unroll 1
    for (int side = 0; side < 2; ++side)
      if (wall(side)) {
        auto value = [&](int k) { return ff2_fma(pw(len - k), B, ff2_fma(pw(k + 1), A, got(k))); };
        const Pair p1 = value(side ? len - 2 : 1);
        Pair s = ff2_fma(T::dup(K.cl[3]), value(side ? len - 3 : 2), T::zero());
        s = ff2_fma(T::dup(K.cl[2]), p1, s);
        s = ff2_fma(T::dup(K.cl[1]), ff2_unpack(W[(4 + side) * L + r]), s);
        W[side * L + r] = ff2_pack(ff2_fma(T::dup(K.cl[0]), ff2_unpack(W[(2 + side) * L + r]), s));
        W[(6 + side) * L + r] = ff2_pack(p1);
      }
    __syncthreads();
    if (act) {
      const Pair wl = ff2_unpack(W[r]), wr = ff2_unpack(W[L + r]), wa = T::dup(K.wa), wb = T::dup(K.wb);
      const Pair Aw = ff2_fma(wb, wr, ff2_fma(wa, wl, T::zero()));
      const Pair Bw = ff2_fma(wb, wl, ff2_fma(wa, wr, T::zero()));
      if (t0 - 2 < K.reach) A = ff2_fma(pw(t0 - 2), Aw, A);
      if (n - t1 - 2 < K.reach) B = ff2_fma(pw(n - t1 - 2), Bw, B);
#pragma unroll 1
      for (int side = 0; side < 2; ++side)
        if (wall(side)) {  // the wall rows: x_0 = R_0 - a_0 x_1
          Pair x1 = ff2_add(ff2_unpack(W[(6 + side) * L + r]), side ? Bw : Aw);
          if (n - 3 < K.reach) x1 = ff2_fma(pw(n - 3), side ? Aw : Bw, x1);
          Pair x0 = ff2_fma(T::dup(K.c0[2]), x1, T::zero());
          x0 = ff2_fma(T::dup(K.c0[1]), ff2_unpack(W[(4 + side) * L + r]), x0);
          W[(6 + side) * L + r] = ff2_pack(ff2_fma(T::dup(K.c0[0]), ff2_unpack(W[(2 + side) * L + r]), x0));
        }
    }
  }
  // x_t = local + A r^(k+1) + B r^(len-k); past `near` points a term only reaches the low part
  if (act) {
    const int near = K.near;
#pragma unroll 1
    for (int k = 0; k < len; ++k) {
      Pair y = got(k);
      const Pair pa = pw(k + 1), pb = pw(len - k);
      if (k + 1 < near) y = ff2_fma_u(pa, A, y);
      else y.lo = v2_fma(pa.hi, A.hi, y.lo);
      if (len - k < near) y = ff2_fma_u(pb, B, y);
      else y.lo = v2_fma(pb.hi, B.hi, y.lo);
      y = ff2_norm(y);
      if (gout) gout[k * gs] = ff2_to_slot(y);
      else col[k * Lp] = ff2_to_slot(y);
    }
    if (wall(0)) gout[0] = ff2_to_slot(ff2_unpack(W[6 * L + r]));
    if (wall(1)) gout[(len - 1) * gs] = ff2_to_slot(ff2_unpack(W[7 * L + r]));
  }
}

// CTA bid: line block bid % nblk of job bid / nblk.  CTAs that run at the same
// time then mostly run the same derivative kind (the instruction cache holds one
// variant), and a field's second read, by the next job, still hits the L2 cache.
template <int LANES>
__device__ __forceinline__ void pair_pass_body(const PairPass& P, unsigned bid) {
  typedef typename Lane<LANES>::Elem Elem;
  if (P.gate && *P.gate) return;
  extern __shared__ __align__(16) float4 pl_smem[];
  const unsigned jb = fdiv(bid, P.divblk), lb = bid - jb * P.nblk;
  const PairJob J = P.job[jb];
  const int n = P.n, L = P.L, Lp = P.Lp, tid = threadIdx.x;
  float4* F = pl_smem;
  Elem* E = (Elem*)(F + (size_t)n * Lp);
  Elem* X = E + P.U * P.nch;
  Elem* W = X + P.U * P.nch;
  Elem* tab = W + 8 * P.U;
  const long long l0 = (long long)lb * L;
  // stage the lines: [t][line]
  for (int idx = tid; idx < n * L; idx += blockDim.x) {
    int t, cl;
    if (P.axis == 0) { cl = (int)fdiv(idx, P.divn); t = idx - cl * n; }
    else { t = (int)fdiv(idx, P.divL); cl = idx - t * L; }
    float4* dst = F + (size_t)t * Lp + cl;
    if (l0 + cl < P.nlines) copy16(dst, J.in + line_start(P, l0 + cl) + (long long)t * P.stride);
    else *dst = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  const float2* gt = (const float2*)P.tab[J.kind];
  for (int i = tid; i < kTab; i += blockDim.x) tab[i] = Lane<LANES>::table(__ldg(gt + i));
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  const int c = (int)fdiv(tid, P.divU), r = tid - c * P.U;
  const long long line = l0 + (LANES == 2 ? r : r >> 1);
  const bool act = c < P.nch && line < P.nlines;
  // strided axes: neighbouring threads hold neighbouring lines, results go straight to global memory
  Elem* gout = nullptr;
  if (P.axis != 0 && act) {
    const long long i = line_start(P, line) + (long long)(c * P.q + min(c, P.rem)) * P.stride;
    gout = (Elem*)(J.out + i) + (LANES == 2 ? 0 : r & 1);
  }
  const long long gs = LANES == 2 ? P.stride : 2 * P.stride;
  if (J.pair_in)  // mixed derivatives: first only
    solve_chunks<LANES, 0, true>(P, (Elem*)F, E, X, W, tab, act, c, r, gout, gs);
  else if (J.kind == 0) solve_chunks<LANES, 0, false>(P, (Elem*)F, E, X, W, tab, act, c, r, gout, gs);
  else solve_chunks<LANES, 1, false>(P, (Elem*)F, E, X, W, tab, act, c, r, gout, gs);
  if (P.axis != 0) return;
  __syncthreads();
  for (int idx = tid; idx < n * L; idx += blockDim.x) {
    const int cl = (int)fdiv(idx, P.divn), t = idx - cl * n;
    if (l0 + cl < P.nlines) J.out[(l0 + cl) * n + t] = F[(size_t)t * Lp + cl];
  }
}

template <int LANES>
__global__ void __launch_bounds__(kMaxThreads, LANES == 2 ? 1 : 2) k_pair_pass(const __grid_constant__ PairPass P) {
  chain_enter();
  pair_pass_body<LANES>(P, blockIdx.x);
}

}  // namespace pl

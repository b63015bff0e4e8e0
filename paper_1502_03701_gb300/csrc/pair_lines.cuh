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
// pointwise map's coefficients carry.
#pragma once
#include "internal.cuh"

namespace pl {

constexpr int kMaxThreads = 512;
constexpr int kTabPow = 72;                    // r^(i - 2), i < kTabPow
constexpr int kTab = kTabPow + kPairMaxC + 1;  // then u0(len), len <= kPairMaxC
constexpr size_t kSmemMax = 200 * 1024;        // dynamic shared memory opt-in

struct PairJob {
  const double* in;  // complex field as reals (pair_in: pairs in the same 8 bytes)
  float2* out;
  int kind;     // 0 first, 1 second derivative
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
  int L, RL, RLp;    // complex lines per CTA, real lines (2 L), shared-memory pitch in reals
  int nch, q, rem;   // chunks per line: the first rem have q + 1 points, the others q
  int bounded;
  FastDiv divblk, divRL, divL, divn, divnx;
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

__device__ __forceinline__ float2 f2(ffn a) { return make_float2(a.hi, a.lo); }

// One chunk of one real line; block-uniform control flow around the barriers.
template <int KIND, bool PAIR>
__device__ __forceinline__ void solve_chunks(const PairPass& P, double* F, float2* E, float2* X, float2* W,
                                             const float2* tab, bool act, int c, int r, float2* gout) {
  const int n = P.n, nch = P.nch, RL = P.RL, RLp = P.RLp;
  const bool bounded = P.bounded;
  const PairKind& K = P.k[KIND];
  auto start_of = [&](int cc) { return cc * P.q + min(cc, P.rem); };
  auto len_of = [&](int cc) { return P.q + (cc < P.rem ? 1 : 0); };
  auto pw = [&](int i) { const float2 v = tab[i + 2]; return ffn{v.x, v.y}; };  // r^i, i >= -2
  const int t0 = act ? start_of(c) : 0, len = act ? len_of(c) : 0, t1 = t0 + len;
  double* col = F + (size_t)t0 * RLp + r;
  auto pairs = [&](int k) -> float2& { return *(float2*)(col + k * RLp); };
  auto got = [&](int k) { const float2 v = pairs(k); return ffn{v.x, v.y}; };
  auto at = [&](int t) -> double {  // staged value at line index t (wrapped, or clamped where it is not used)
    if (bounded) t = min(max(t, 0), n - 1);
    else t = t < 0 ? t + n : (t >= n ? t - n : t);
    return F[(size_t)t * RLp + r];
  };
  auto dif = [&](double a, double b) -> ffn {  // a - b
    if constexpr (PAIR) {
      const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
      return ff2_add(ffn{__int_as_float((int)x), __int_as_float((int)(x >> 32))},
                     ffn{-__int_as_float((int)y), -__int_as_float((int)(y >> 32))});
    } else {
      return ff2_split(a - b);
    }
  };
  auto neg = [](ffn a) { return ffn{-a.hi, -a.lo}; };
  // the neighbours' points, and the wall rows' right-hand sides, before any point is overwritten
  double fm2 = 0, fm1 = 0, fp0 = 0, fp1 = 0;
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
      ffn u, v;
      if (KIND == 0) {
        const int i = side ? n - 2 : 1, k = side ? n - 2 : 0;
        u = dif(at(i + 1), at(i - 1));
        v = dif(at(k + 1), at(k));
      } else {
        auto second = [&](int i) { return ff2_add(dif(at(i + 1), at(i)), neg(dif(at(i), at(i - 1)))); };
        u = second(side ? n - 2 : 1);
        v = second(side ? n - 3 : 2);
      }
      W[(2 + side) * RL + r] = f2(u);
      W[(4 + side) * RL + r] = f2(v);
    }
  __syncthreads();
  // forward sweep from zero, in place: g_t = w_t + r g_{t-1}, w_t = d_t + rho (d_{t-1} + d_{t+1}),
  // d_t = f_{t+1} - f_{t-1} (first) or f_{t+1} - 2 f_t + f_{t-1} (second derivative)
  if (act) {
    double fa = col[0], fb = col[RLp];  // f_t, f_{t+1}
    ffn dm, d, gl{0, 0};
    if (KIND == 0) {
      dm = dif(fa, fm2);
      d = dif(fb, fm1);
    } else {
      const ffn g0 = dif(fm1, fm2), g1 = dif(fa, fm1);
      gl = dif(fb, fa);  // f_{t+1} - f_t
      dm = ff2_add(g1, neg(g0));
      d = ff2_add(gl, neg(g1));
    }
    ffn g{0, 0};
    auto step = [&](int k, double fc) {  // fc = f_{t+2}
      ffn dn;
      if (KIND == 0) {
        dn = dif(fc, fa);
      } else {
        const ffn gn = dif(fc, fb);
        dn = ff2_add(gn, neg(gl));
        gl = gn;
      }
      ffn w = ff2_fma_u(K.rho, ff2_add_u(dm, dn), d);
      if (bounded) {
        const int t = t0 + k;
        if (t < 2 || t > n - 3) w = ffn{0, 0};
      }
      g = ff2_fma(K.r, g, w);
      pairs(k) = f2(g);
      dm = d;
      d = dn;
      fa = fb;
      fb = fc;
    };
#pragma unroll 2
    for (int k = 0; k < len; ++k) step(k, k + 2 < len ? col[(k + 2) * RLp] : k + 2 == len ? fp0 : fp1);
    E[c * RL + r] = f2(g);
  }
  __syncthreads();
  // the true g at the point before the chunk
  ffn G{0, 0};
  if (act) {
    int off = 0, cc = c;
    for (int j = 0; j < nch && off < K.reach; ++j) {
      if (--cc < 0) {
        if (bounded) break;
        cc += nch;
      }
      const float2 e = E[cc * RL + r];
      G = ff2_fma(pw(off), ffn{e.x, e.y}, G);
      off += len_of(cc);
    }
    if (!bounded && n < K.reach) G = ff2_fma(K.invn, G, ffn{0, 0});  // the line closes on itself
    // backward sweep from zero, in place: x_t = g_t + r x_{t+1}
    ffn x{0, 0};
#pragma unroll 4
    for (int k = len - 1; k >= 0; --k) {
      x = ff2_fma(K.r, x, got(k));
      pairs(k) = f2(x);
    }
    const float2 u0 = tab[kTabPow + len];
    X[c * RL + r] = f2(ff2_fma(ffn{u0.x, u0.y}, G, x));
  }
  __syncthreads();
  ffn A{0, 0}, B{0, 0};
  if (act) {
    ffn xn{0, 0};  // the true x at the point after the chunk
    int off = 0, cc = c;
    for (int j = 0; j < nch && off < K.reach; ++j) {
      if (++cc >= nch) {
        if (bounded) break;
        cc -= nch;
      }
      const float2 e = X[cc * RL + r];
      xn = ff2_fma(pw(off), ffn{e.x, e.y}, xn);
      off += len_of(cc);
    }
    if (!bounded && n < K.reach) xn = ff2_fma(K.invn, xn, ffn{0, 0});
    A = ff2_fma(K.kap, G, ffn{0, 0});
    B = ff2_fma(neg(pw(len + 1)), A, xn);
  }
  if (bounded) {
    auto load = [](const float2* p) { const float2 x = *p; return ffn{x.x, x.y}; };
#pragma unroll 1
    for (int side = 0; side < 2; ++side)
      if (wall(side)) {
        auto value = [&](int k) { return ff2_fma(pw(len - k), B, ff2_fma(pw(k + 1), A, got(k))); };
        const ffn p1 = value(side ? len - 2 : 1);
        ffn s = ff2_fma(K.cl[3], value(side ? len - 3 : 2), ffn{0, 0});
        s = ff2_fma(K.cl[2], p1, s);
        s = ff2_fma(K.cl[1], load(W + (4 + side) * RL + r), s);
        W[side * RL + r] = f2(ff2_fma(K.cl[0], load(W + (2 + side) * RL + r), s));
        W[(6 + side) * RL + r] = f2(p1);
      }
    __syncthreads();
    if (act) {
      const ffn wl = load(W + r), wr = load(W + RL + r);
      const ffn Aw = ff2_fma(K.wb, wr, ff2_fma(K.wa, wl, ffn{0, 0}));
      const ffn Bw = ff2_fma(K.wb, wl, ff2_fma(K.wa, wr, ffn{0, 0}));
      if (t0 - 2 < K.reach) A = ff2_fma(pw(t0 - 2), Aw, A);
      if (n - t1 - 2 < K.reach) B = ff2_fma(pw(n - t1 - 2), Bw, B);
#pragma unroll 1
      for (int side = 0; side < 2; ++side)
        if (wall(side)) {  // the wall rows: x_0 = R_0 - a_0 x_1
          ffn x1 = ff2_add(load(W + (6 + side) * RL + r), side ? Bw : Aw);
          if (n - 3 < K.reach) x1 = ff2_fma(pw(n - 3), side ? Aw : Bw, x1);
          ffn x0 = ff2_fma(K.c0[1], load(W + (4 + side) * RL + r), ff2_fma(K.c0[2], x1, ffn{0, 0}));
          W[(6 + side) * RL + r] = f2(ff2_fma(K.c0[0], load(W + (2 + side) * RL + r), x0));
        }
    }
  }
  // x_t = local + A r^(k+1) + B r^(len-k); past `near` points a term only reaches the low part
  if (act) {
    const int near = K.near;
    const long long gs = 2 * P.stride;
#pragma unroll 1
    for (int k = 0; k < len; ++k) {
      ffn y = got(k);
      const ffn pa = pw(k + 1), pb = pw(len - k);
      if (k + 1 < near) y = ff2_fma_u(pa, A, y);
      else y.lo = __fmaf_rn(pa.hi, A.hi, y.lo);
      if (len - k < near) y = ff2_fma_u(pb, B, y);
      else y.lo = __fmaf_rn(pb.hi, B.hi, y.lo);
      y = ff2_norm(y);
      if (gout) gout[k * gs] = f2(y);
      else pairs(k) = f2(y);
    }
    if (wall(0)) gout[0] = W[6 * RL + r];
    if (wall(1)) gout[(len - 1) * gs] = W[7 * RL + r];
  }
}

// CTA bid: line block bid % nblk of job bid / nblk.  CTAs that run at the same
// time then mostly run the same derivative kind (the instruction cache holds one
// variant), and a field's second read, by the next job, still hits the L2 cache.
__device__ __forceinline__ void pair_pass_body(const PairPass& P, unsigned bid) {
  if (P.gate && *P.gate) return;
  extern __shared__ __align__(16) double pl_smem[];
  const unsigned jb = fdiv(bid, P.divblk), lb = bid - jb * P.nblk;
  const PairJob J = P.job[jb];
  const int n = P.n, L = P.L, RL = P.RL, RLp = P.RLp, tid = threadIdx.x;
  double* F = pl_smem;
  float2* E = (float2*)(F + (size_t)n * RLp);
  float2* X = E + RL * P.nch;
  float2* W = X + RL * P.nch;
  float2* tab = W + 8 * RL;
  const long long l0 = (long long)lb * L;
  // stage the lines: [t][line][re, im]
  for (int idx = tid; idx < n * L; idx += blockDim.x) {
    int t, cl;
    if (P.axis == 0) { cl = (int)fdiv(idx, P.divn); t = idx - cl * n; }
    else { t = (int)fdiv(idx, P.divL); cl = idx - t * L; }
    double* dst = F + (size_t)t * RLp + 2 * cl;
    if (l0 + cl < P.nlines) copy16(dst, J.in + 2 * (line_start(P, l0 + cl) + (long long)t * P.stride));
    else *(double2*)dst = make_double2(0.0, 0.0);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  const float2* gt = (const float2*)P.tab[J.kind];
  for (int i = tid; i < kTab; i += blockDim.x) tab[i] = __ldg(gt + i);
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  const int c = (int)fdiv(tid, P.divRL), r = tid - c * RL;
  const bool act = c < P.nch && l0 + (r >> 1) < P.nlines;
  // strided axes: neighbouring threads hold neighbouring reals, results go straight to global memory
  float2* gout = nullptr;
  if (P.axis != 0 && act) {
    const int t0 = c * P.q + min(c, P.rem);
    gout = J.out + 2 * (line_start(P, l0 + (r >> 1)) + (long long)t0 * P.stride) + (r & 1);
  }
  if (J.pair_in) solve_chunks<0, true>(P, F, E, X, W, tab, act, c, r, gout);  // mixed derivatives: first only
  else if (J.kind == 0) solve_chunks<0, false>(P, F, E, X, W, tab, act, c, r, gout);
  else solve_chunks<1, false>(P, F, E, X, W, tab, act, c, r, gout);
  if (P.axis != 0) return;
  __syncthreads();
  for (int idx = tid; idx < n * L; idx += blockDim.x) {
    const int cl = (int)fdiv(idx, P.divn), t = idx - cl * n;
    if (l0 + cl < P.nlines) {
      const float4 v = *(const float4*)(F + (size_t)t * RLp + 2 * cl);
      *(float4*)(J.out + 2 * ((l0 + cl) * n + t)) = v;
    }
  }
}

__global__ void __launch_bounds__(kMaxThreads, 2) k_pair_pass(const __grid_constant__ PairPass P) {
  pair_pass_body(P, blockIdx.x);
}

}  // namespace pl

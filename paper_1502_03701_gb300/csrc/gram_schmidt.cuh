// Gram-Schmidt device code shared by the Krylov kernels and the GMRES cycle.
#pragma once
#include <cuda_runtime.h>

#include "pairs.cuh"

namespace gs {

__device__ __forceinline__ double warp_sum(double x) {
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// ---------------------------------------------------------------------------
// Gram-Schmidt passes for up to kColMax basis vectors: V^H w (dots), w -= V h
// (update), or both with one read of V.
//
// What bounds them: the basis is read from HBM once per pass, 16 bytes and
// about 60 FP32 issue slots per entry (FP64 runs at 1/64 of the FP32 rate, so
// products are exact FP32 two-products of split pairs on the packed FP32
// instructions).  A CTA of 16 warps takes 32 RG rows at a time: the warps of a
// row group (CW of them, up to four columns each) hold the group's part of V in
// registers as pairs, add up w's correction, exchange it through shared memory
// and take the new w's products with the same registers, so the second pass of
// CGS2 reads V once and splits it once.  The next rows' loads are in flight
// meanwhile.  Sums over blocks: the last block to finish adds the blocks'
// partial sums in block order (reproducible) and resets the counter.
// 524,288 unknowns, 55 vectors: the three passes of CGS2 take 139, 226 and 108 us
// (481 MB each, 62 to 66 % of the issue slots; 164, 387 and 273 us as kernels of
// one warp per column and FP64 every fourth column, with V read twice).
// ---------------------------------------------------------------------------
constexpr int kColThreads = 512, kColWarps = kColThreads / 32, kCpw = 4, kColMax = kColWarps * kCpw;

// column warps per row group: the smallest power of two with kCpw CW >= k
__host__ __device__ inline int col_warps(int k) {
  int cw = 1;
  while (cw * kCpw < k) cw *= 2;
  return cw;
}
// One row per thread from 384 rows per SM up, for more columns than a warp holds.  Up to four columns stay with the
// column split at every size: a row's columns are then in one warp, so it reads V once with no barrier in the loop.
// CGS2 of 4,194,304 unknowns against 1, 2 and 4 vectors 223, 252 and 295 us (320, 390 and 479 one row per thread),
// of 10,485,760 against 1 and 4 482 and 665 us (726 and 1,130), of 131,072 against 4 54 us (57).
__host__ __device__ inline bool by_rows(long long n, int k) { return n >= 152LL * 384 && k > kCpw; }
inline int col_blocks(long long n, int k) {
  if (by_rows(n, k)) return 152;
  const long long rows = 32LL * (kColWarps / col_warps(k));
  const long long b = (n + rows - 1) / rows;
  return (int)(b < 152 ? (b < 1 ? 1 : b) : 152);
}

struct ColArgs {
  const double2* V;
  double2* w;
  const double2* h;     // update: coefficients (null: none)
  double2* partial;     // dots: nb x k block sums (null: none)
  double* npart;        // |w|^2 block sums (null: none)
  double2* out_h;       // dots: the reduced sums
  double2* sum_h;       // added to as well when set (h1 + h2)
  double* out_norm;     // ||w|| (of the updated w)
  double* ref_norm;     // decide: ||w|| before the update; *skip = out >= eta ref
  int* skip;
  unsigned* counter;    // zero on entry, zero on exit
  long long n;
  int k, nb;
};

struct ColShared {
  float4 H[kColMax][2];       // coefficients as duplicated pairs, re and im
  union {
    struct {
      float4 red[kColWarps][32];  // column split: a warp's share of the correction per row, pairs re, im
      float4 wn[kColWarps][32][2];  // the group's updated w as duplicated pairs, re and im
    };
    struct {
      float4 wr[kColThreads], wi[kColThreads];  // row split: the chunk's w as duplicated pairs
    };
  };
  double2 dots[kColWarps][kCpw];
  double nrm[kColWarps];
  int last;
};

// hi, lo of a complex value as one packed pair (re, im), and one component duplicated
__device__ __forceinline__ ffn2 dup_part(ffn2 a, bool im) {
  return im ? ffn2{v2(a.hi.y), v2(a.lo.y)} : ffn2{v2(a.hi.x), v2(a.lo.x)};
}
__device__ __forceinline__ ffn2 swap_parts(ffn2 a) {
  return ffn2{make_float2(a.hi.y, a.hi.x), make_float2(a.lo.y, a.lo.x)};
}

// A warp's column sums and norm into shared memory.
template <bool DOTS, bool NORM>
__device__ __forceinline__ void warp_sums(const ColArgs& A, ColShared& S, ffn2* d1, ffn2* d2, double nrm) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // block sums
  if (DOTS) {
    // the four columns' sums over the lanes together: the first two steps halve the columns that a
    // lane carries, so six exchanges serve all of them; lanes 0, 8, 16, 24 end with columns 0..3
    ffn2 t[kCpw];
#pragma unroll
    for (int q = 0; q < kCpw; ++q) {
      ffn2 a = d1[q];
      a.hi.y = -a.hi.y;
      a.lo.y = -a.lo.y;
      t[q] = ff2_add(a, swap_parts(d2[q]));  // (d1.re + d2.im, d2.re - d1.im)
    }
    auto other = [](ffn2 x, int o) {
      return ffn2{make_float2(__shfl_xor_sync(0xffffffffu, x.hi.x, o), __shfl_xor_sync(0xffffffffu, x.hi.y, o)),
                  make_float2(__shfl_xor_sync(0xffffffffu, x.lo.x, o), __shfl_xor_sync(0xffffffffu, x.lo.y, o))};
    };
    auto choose = [](bool c, ffn2 x, ffn2 y) { return c ? x : y; };
    const bool up = lane & 16, mid = lane & 8;
    const ffn2 u0 = ff2_add(choose(up, t[2], t[0]), other(choose(up, t[0], t[2]), 16));
    const ffn2 u1 = ff2_add(choose(up, t[3], t[1]), other(choose(up, t[1], t[3]), 16));
    ffn2 v = ff2_add(choose(mid, u1, u0), other(choose(mid, u0, u1), 8));
    for (int o = 4; o > 0; o >>= 1) v = ff2_add(v, other(v, o));
    if ((lane & 7) == 0) S.dots[wid][lane >> 3] = ff2_to_d(v);
  }
  if (NORM) {
    nrm = warp_sum(nrm);
    if (lane == 0) S.nrm[wid] = nrm;
  }
  __syncthreads();
}

// this block's sum of column j over its row groups
__device__ __forceinline__ double2 block_dot(const ColShared& S, int j, int CW) {
  const int c = j % CW, q = j / CW;
  double sr = 0.0, si = 0.0;
  for (int g = 0; g < kColWarps / CW; ++g) {
    sr += S.dots[g * CW + c][q].x;
    si += S.dots[g * CW + c][q].y;
  }
  return make_double2(sr, si);
}
// this block's |w|^2 from every step-th warp
__device__ __forceinline__ double block_nrm(const ColShared& S, int step) {
  double t = 0.0;
  for (int g = 0; g < kColWarps; g += step) t += S.nrm[g];
  return t;
}

template <bool UPDATE, bool DOTS, bool NORM>
__device__ __forceinline__ void finish_pass(const ColArgs& A, unsigned bidx, ColShared& S, ffn2* d1, ffn2* d2,
                                            double nrm) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, k = A.k;
  warp_sums<DOTS, NORM>(A, S, d1, d2, nrm);
  if (DOTS && threadIdx.x < k) A.partial[(long long)bidx * k + threadIdx.x] = block_dot(S, threadIdx.x, col_warps(k));
  if (NORM && threadIdx.x == kColThreads - 1) A.npart[bidx] = block_nrm(S, 1);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) S.last = atomicAdd(A.counter, 1u) == (unsigned)A.nb - 1;
  __syncthreads();
  if (!S.last) return;
  __threadfence();
  if (DOTS) {
    for (int j = wid; j < k; j += kColWarps) {
      double sr = 0.0, si = 0.0;
#pragma unroll 5
      for (int b = lane; b < A.nb; b += 32) {
        const double2 p = __ldcg(A.partial + (long long)b * k + j);
        sr += p.x;
        si += p.y;
      }
      sr = warp_sum(sr);
      si = warp_sum(si);
      if (lane == 0) {
        A.out_h[j] = make_double2(sr, si);
        if (A.sum_h) A.sum_h[j] = make_double2(A.sum_h[j].x + sr, A.sum_h[j].y + si);
      }
    }
  }
  if (NORM && wid == kColWarps - 1) {
    double t = 0.0;
#pragma unroll 5
    for (int b = lane; b < A.nb; b += 32) t += __ldcg(A.npart + b);
    t = sqrt(warp_sum(t));
    if (lane == 0) {
      *A.out_norm = t;
      if (A.skip) *A.skip = t >= 0.70710678118654752 * *A.ref_norm;  // NaN: reorthogonalise (and let the norm report it)
    }
  }
  if (UPDATE && !DOTS && A.sum_h)
    for (int j = threadIdx.x; j < k; j += kColThreads)
      A.sum_h[j] = make_double2(A.sum_h[j].x + A.h[j].x, A.sum_h[j].y + A.h[j].y);
  if (threadIdx.x == 0) *A.counter = 0u;
}

// the coefficients as duplicated pairs in shared memory
__device__ __forceinline__ void put_coef(ColShared& S, int j, double2 h) {
  const ffn2 p = ff2_split(h);
  S.H[j][0] = ff2_pack(dup_part(p, false));
  S.H[j][1] = ff2_pack(dup_part(p, true));
}
__device__ __forceinline__ void load_coefs(const double2* h, int k, ColShared& S) {
  for (int j = threadIdx.x; j < k; j += kColThreads) put_coef(S, j, h[j]);
  __syncthreads();
}

// The rows of block bidx of A.nb, columns split over the warps.  coefs() fills
// S.H (update only) while the first rows' loads are in flight.
template <bool UPDATE, bool DOTS, bool NORM, class Coefs>
__device__ __forceinline__ void col_main(const ColArgs& A, unsigned bidx, ColShared& S, ffn2* d1, ffn2* d2,
                                         double& nrm, Coefs coefs) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int k = A.k, CW = col_warps(k), RG = kColWarps / CW;
  const int grp = wid / CW, cw = wid - grp * CW;
  const long long n = A.n;
  // conj(V_j) w = d1.re + d2.im, d2.re - d1.im with d1 += V_j re(w), d2 += V_j im(w)
#pragma unroll
  for (int q = 0; q < kCpw; ++q) d1[q] = d2[q] = ff2_zero2();
  nrm = 0.0;
  const long long step = 32LL * RG * A.nb;
  long long row = 32LL * ((long long)bidx * RG + grp) + lane;
  double2 nv[kCpw], nw = make_double2(0.0, 0.0);
  auto fetch = [&](long long r) {
#pragma unroll
    for (int q = 0; q < kCpw; ++q) {
      const int j = cw + q * CW;
      nv[q] = j < k && r < n ? A.V[(long long)j * n + r] : make_double2(0.0, 0.0);
    }
    if (!UPDATE || cw == 0) nw = r < n ? A.w[r] : make_double2(0.0, 0.0);
  };
  fetch(row);
  if (UPDATE) coefs();
  int rounds = 0;
  for (long long r0 = 32LL * bidx * RG; r0 < n; r0 += step, row += step) {  // block-uniform
    ffn2 v[kCpw];
    const double2 wold = nw;
#pragma unroll
    for (int q = 0; q < kCpw; ++q) v[q] = ff2_split(nv[q]);
    fetch(row + step);
    ffn2 wr, wi;
    if (UPDATE) {
      // V h = a1 + i a2 with a1 += V re(h), a2 += V im(h)
      ffn2 a1 = ff2_zero2(), a2 = ff2_zero2();
#pragma unroll
      for (int q = 0; q < kCpw; ++q) {
        const int j = cw + q * CW;
        if (j < k) {
          a1 = ff2_fma_u(ff2_unpack(S.H[j][0]), v[q], a1);
          a2 = ff2_fma_u(ff2_unpack(S.H[j][1]), v[q], a2);
        }
      }
      ffn2 s2 = swap_parts(a2);  // i a2 = (-im, re)
      s2.hi.x = -s2.hi.x;
      s2.lo.x = -s2.lo.x;
      const ffn2 mine = ff2_add(a1, s2);
      if (CW > 1) {
        S.red[wid][lane] = ff2_pack(mine);
        __syncthreads();
      }
      if (cw == 0) {
        ffn2 t = mine;
        for (int c = 1; c < CW; ++c) t = ff2_add(t, ff2_unpack(S.red[wid + c][lane]));
        const double2 wnew = make_double2(wold.x - ff2_to_d(ffn{t.hi.x, t.lo.x}), wold.y - ff2_to_d(ffn{t.hi.y, t.lo.y}));
        if (row < n) A.w[row] = wnew;
        if (NORM) nrm = fma(wnew.x, wnew.x, fma(wnew.y, wnew.y, nrm));
        if (DOTS) {
          const ffn2 p = ff2_split(wnew);
          wr = dup_part(p, false);
          wi = dup_part(p, true);
          if (CW > 1) {
            S.wn[grp][lane][0] = ff2_pack(wr);
            S.wn[grp][lane][1] = ff2_pack(wi);
          }
        }
      }
      if (CW > 1) {
        __syncthreads();
        if (DOTS && cw != 0) {
          wr = ff2_unpack(S.wn[grp][lane][0]);
          wi = ff2_unpack(S.wn[grp][lane][1]);
        }
      }
    } else {
      const ffn2 p = ff2_split(wold);
      wr = dup_part(p, false);
      wi = dup_part(p, true);
      if (NORM && cw == 0) nrm = fma(wold.x, wold.x, fma(wold.y, wold.y, nrm));
    }
    if (DOTS) {
#pragma unroll
      for (int q = 0; q < kCpw; ++q)
        if (cw + q * CW < k) {
          d1[q] = ff2_fma_u(wr, v[q], d1[q]);
          d2[q] = ff2_fma_u(wi, v[q], d2[q]);
        }
      if ((++rounds & 3) == 0) {
#pragma unroll
        for (int q = 0; q < kCpw; ++q) {
          d1[q] = ff2_norm(d1[q]);
          d2[q] = ff2_norm(d2[q]);
        }
      }
    }
  }
}

template <bool UPDATE, bool DOTS, bool NORM>
__device__ __forceinline__ void col_pass(const ColArgs& A, unsigned bidx, ColShared& S) {
  ffn2 d1[kCpw], d2[kCpw];
  double nrm;
  col_main<UPDATE, DOTS, NORM>(A, bidx, S, d1, d2, nrm, [&]() { load_coefs(A.h, A.k, S); });
  finish_pass<UPDATE, DOTS, NORM>(A, bidx, S, d1, d2, nrm);
}

// The same passes with one row per thread in the update (no exchange between
// warps) and the products column by column afterwards: the chunk of V that the
// update has just read (512 rows; 68 MB over all SMs at k = 55) comes back from
// L2.  Needs enough rows to fill the threads.  With the column split, the
// exchange of 16 warps' shares per 32 rows left 60 % of the issue slots empty at
// k = 55 (312 us for update + products of 524,288 unknowns).
template <bool UPDATE, bool DOTS, bool NORM>
__device__ __forceinline__ void row_pass(const ColArgs& A, unsigned bidx, ColShared& S) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int k = A.k, CW = col_warps(k), RG = kColWarps / CW;
  const int grp = wid / CW, cw = wid - grp * CW;
  const long long n = A.n;
  if (UPDATE) load_coefs(A.h, k, S);
  ffn2 d1[kCpw], d2[kCpw];
#pragma unroll
  for (int q = 0; q < kCpw; ++q) d1[q] = d2[q] = ff2_zero2();
  double nrm = 0.0;
  int rounds = 0;  // over all chunks: with few columns a warp has one or two rounds of each
  const long long rows = ((n + A.nb - 1) / A.nb + 31) / 32 * 32;
  const long long r0 = rows * bidx, r1 = r0 + rows < n ? r0 + rows : n;
  for (long long c0 = r0; c0 < r1; c0 += kColThreads) {
    const long long row = c0 + threadIdx.x;
    double2 w = make_double2(0.0, 0.0);
    if (row < r1) {
      w = A.w[row];
      if (UPDATE) {
        const double2* Vr = A.V + row;
        ffn2 a1 = ff2_zero2(), a2 = ff2_zero2();
        constexpr int G = 4;  // columns per step, the next step's in flight
        double2 v[G], nx[G];
        auto fetch = [&](int j0) {
#pragma unroll
          for (int q = 0; q < G; ++q)
            if (j0 + q < k) nx[q] = Vr[(long long)(j0 + q) * n];
        };
        fetch(0);
        for (int j0 = 0; j0 < k; j0 += G) {
#pragma unroll
          for (int q = 0; q < G; ++q) v[q] = nx[q];
          fetch(j0 + G);
#pragma unroll
          for (int q = 0; q < G; ++q) {
            if (j0 + q >= k) break;
            const ffn2 p = ff2_split(v[q]);
            a1 = ff2_fma_u(ff2_unpack(S.H[j0 + q][0]), p, a1);
            a2 = ff2_fma_u(ff2_unpack(S.H[j0 + q][1]), p, a2);
          }
          a1 = ff2_norm(a1);
          a2 = ff2_norm(a2);
        }
        ffn2 s2 = swap_parts(a2);  // i a2 = (-im, re)
        s2.hi.x = -s2.hi.x;
        s2.lo.x = -s2.lo.x;
        const double2 c = ff2_to_d(ff2_add(a1, s2));
        w = make_double2(w.x - c.x, w.y - c.y);
        A.w[row] = w;
      }
      if (NORM) nrm = fma(w.x, w.x, fma(w.y, w.y, nrm));
    }
    if (DOTS) {
      const ffn2 p = ff2_split(w);
      S.wr[threadIdx.x] = ff2_pack(dup_part(p, false));
      S.wi[threadIdx.x] = ff2_pack(dup_part(p, true));
      __syncthreads();
      const int per = kColThreads / RG;  // rows of this warp's group
      const int left = (int)(r1 - c0 < kColThreads ? r1 - c0 : kColThreads);
      const int i1 = grp * per + per < left ? grp * per + per : left;
      double2 v[kCpw], nx[kCpw];
      auto fetch = [&](int i) {
#pragma unroll
        for (int q = 0; q < kCpw; ++q) {
          const int j = cw + q * CW;
          nx[q] = i + lane < i1 && j < k ? A.V[(long long)j * n + c0 + i + lane] : make_double2(0.0, 0.0);
        }
      };
      fetch(grp * per);
      for (int i = grp * per; i < i1; i += 32) {
#pragma unroll
        for (int q = 0; q < kCpw; ++q) v[q] = nx[q];
        fetch(i + 32);
        const ffn2 wr = ff2_unpack(S.wr[i + lane]), wi = ff2_unpack(S.wi[i + lane]);
#pragma unroll
        for (int q = 0; q < kCpw; ++q)
          if (cw + q * CW < k) {
            const ffn2 p = ff2_split(v[q]);
            d1[q] = ff2_fma_u(wr, p, d1[q]);
            d2[q] = ff2_fma_u(wi, p, d2[q]);
          }
        if ((++rounds & 3) == 0) {
#pragma unroll
          for (int q = 0; q < kCpw; ++q) {
            d1[q] = ff2_norm(d1[q]);
            d2[q] = ff2_norm(d2[q]);
          }
        }
      }
      __syncthreads();
    }
  }
  finish_pass<UPDATE, DOTS, NORM>(A, bidx, S, d1, d2, nrm);
}

// ---------------------------------------------------------------------------
// CGS2 of small vectors with the column sums added up inside clusters of CTAs,
// through distributed shared memory.  Below 16,384 unknowns the passes are
// latency, not bandwidth: with sums through global memory and a last block's
// reduction they took 39 us for 8,192 unknowns and 20 vectors, most of it fences,
// atomics and the reduction of 128 partial sums per column.
//  - up to kCluOneN unknowns one cluster of 16 takes all rows and all three
//    passes in one launch;
//  - above, three launches of up to 16 clusters of 8 (of clusters of 16 the
//    device holds too few at a time); every cluster leaves one partial sum per
//    column and the next launch adds these up: 29 us for those 8,192 unknowns.
// Where the lines lie (stab_orthogonalize, with about 40 us of copy and wait):
// 2,048 unknowns 43 us in one launch and 55 in three for 8 vectors, 51 and 55 for
// 29; 3,072 unknowns 58 and 55 for 29 vectors, 78 and 55 for 55.  15,360 unknowns,
// 29 vectors: 71 us in clusters, 80 with sums through global memory.
// ---------------------------------------------------------------------------
constexpr int kCluOne = 16, kClu = 8, kCluMax = 16;  // CTAs per cluster (one launch, passes), clusters
constexpr long long kCluOneN = 2048;   // one cluster in one launch up to here
constexpr long long kCluMaxN = 16384;  // passes in clusters below

__host__ __device__ inline int clu_count(long long n, int k) {
  const long long rows = 32LL * (kColWarps / col_warps(k)) * kClu, c = (n + rows - 1) / rows;
  return (int)(c < kCluMax ? c : kCluMax);
}

struct CluShared {
  ColShared S;
  double2 part[2][kColMax];  // this CTA's column sums (two buffers: a pass may start while others still read)
  double2 h[2][kColMax];     // coefficients of the two passes
  double npart, norm;
};

struct CluArgs {
  const double2* V;
  double2* w;
  double2* p1;     // clusters x k column sums of the first pass
  double2* p2;     // of the second
  double2* d_h;    // h1 + h2
  double* np;      // |w|^2 per cluster
  double* d_norm;  // ||w||
  unsigned* counter;
  long long n;
  int k, G;  // vectors, clusters
};

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
// the value at shared-memory address p of CTA `rank` of the cluster
__device__ __forceinline__ double cluster_load(const double* p, unsigned rank) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  unsigned r;
  double v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(r) : "memory");
  return v;
}

// Sums of the CTAs' column sums to put(j, sum), ranks in a fixed tree; this CTA takes the columns
// j0, j0 + dj, ...: CLU lanes per column.
template <int CLU, class Put>
__device__ __forceinline__ void cluster_dots(CluShared& C, int buf, int k, int j0, int dj, Put put) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, sub = lane / CLU, rank = lane % CLU;
  constexpr int PER = 32 / CLU;  // columns per warp
  if (threadIdx.x < k) C.part[buf][threadIdx.x] = block_dot(C.S, threadIdx.x, col_warps(k));
  cluster_barrier();
  for (int jj = j0 + PER * wid * dj; jj < k; jj += PER * kColWarps * dj) {  // warp-uniform
    const int j = jj + sub * dj;
    double x = 0.0, y = 0.0;
    if (j < k) {
      x = cluster_load(&C.part[buf][j].x, rank);
      y = cluster_load(&C.part[buf][j].y, rank);
    }
    for (int o = CLU / 2; o > 0; o >>= 1) {
      x += __shfl_xor_sync(0xffffffffu, x, o);
      y += __shfl_xor_sync(0xffffffffu, y, o);
    }
    if (j < k && rank == 0) put(j, make_double2(x, y));
  }
}

__device__ __forceinline__ ColArgs clu_rows(const CluArgs& A, int ctas) {
  ColArgs P{};
  P.V = A.V;
  P.w = A.w;
  P.k = A.k;
  P.n = A.n;
  P.nb = ctas;
  return P;
}

// The whole CGS2 in one cluster; every CTA returns with C.norm = ||w||.  To be followed by cluster_barrier():
// a CTA may not exit while others read its shared memory.
__device__ __forceinline__ void cgs2_cluster(const CluArgs& A, unsigned rank, CluShared& C) {
  const ColArgs P = clu_rows(A, kCluOne);
  const int k = A.k;
  ffn2 d1[kCpw], d2[kCpw];
  double nrm;
  col_main<false, true, false>(P, rank, C.S, d1, d2, nrm, []() {});
  warp_sums<true, false>(P, C.S, d1, d2, nrm);
  cluster_dots<kCluOne>(C, 0, k, 0, 1, [&](int j, double2 h) { C.h[0][j] = h; });
  __syncthreads();
  col_main<true, true, false>(P, rank, C.S, d1, d2, nrm, [&]() { load_coefs(C.h[0], k, C.S); });
  warp_sums<true, false>(P, C.S, d1, d2, nrm);
  cluster_dots<kCluOne>(C, 1, k, 0, 1, [&](int j, double2 h) { C.h[1][j] = h; });
  __syncthreads();
  if (rank == 0 && threadIdx.x < k) {
    const double2 a = C.h[0][threadIdx.x], b = C.h[1][threadIdx.x];
    A.d_h[threadIdx.x] = make_double2(a.x + b.x, a.y + b.y);
  }
  col_main<true, false, true>(P, rank, C.S, d1, d2, nrm, [&]() { load_coefs(C.h[1], k, C.S); });
  warp_sums<false, true>(P, C.S, d1, d2, nrm);
  if (threadIdx.x == 0) C.npart = block_nrm(C.S, col_warps(k));  // a row group's first warp has its rows
  cluster_barrier();
  if (threadIdx.x < 32) {
    double t = threadIdx.x < kCluOne ? cluster_load(&C.npart, threadIdx.x) : 0.0;
    t = sqrt(warp_sum(t));
    if (threadIdx.x == 0) {
      C.norm = t;
      if (rank == 0) *A.d_norm = t;
    }
  }
  __syncthreads();
}

// One pass (0: h1 = V^H w, 1: w -= V h1 and h2 = V^H w, 2: w -= V h2 and ||w||) of CTA `rank` of cluster g.
template <int PASS>
__device__ __forceinline__ void cgs2_clusters(const CluArgs& A, unsigned g, unsigned rank, CluShared& C) {
  const ColArgs P = clu_rows(A, kClu * A.G);
  const int k = A.k, t = threadIdx.x;
  // the sum over the clusters, half of them on each of two neighbouring lanes
  auto total = [&](const double2* p, int j, int half) {
    double2 v[kCluMax / 2], s = make_double2(0.0, 0.0);
#pragma unroll
    for (int q = 0; q < kCluMax / 2; ++q) {
      const int g = q + half * (kCluMax / 2);
      v[q] = g < A.G && j < k ? p[g * k + j] : make_double2(0.0, 0.0);
    }
#pragma unroll
    for (int q = 0; q < kCluMax / 2; ++q) {
      s.x += v[q].x;
      s.y += v[q].y;
    }
    return make_double2(s.x + __shfl_xor_sync(0xffffffffu, s.x, 1), s.y + __shfl_xor_sync(0xffffffffu, s.y, 1));
  };
  ffn2 d1[kCpw], d2[kCpw];
  double nrm;
  col_main<PASS != 0, PASS != 2, PASS == 2>(P, g * kClu + rank, C.S, d1, d2, nrm, [&]() {
    if (t < 2 * kColMax) {  // whole warps
      const int j = t >> 1;
      const double2 h = total(PASS == 1 ? A.p1 : A.p2, j, t & 1);
      if (j < k && !(t & 1)) put_coef(C.S, j, h);
      if (PASS == 2 && g == 0 && rank == 0) {
        const double2 h1 = total(A.p1, j, t & 1);
        if (j < k && !(t & 1)) A.d_h[j] = make_double2(h1.x + h.x, h1.y + h.y);
      }
    }
    __syncthreads();
  });
  warp_sums<PASS != 2, PASS == 2>(P, C.S, d1, d2, nrm);
  if (PASS != 2) {
    double2* out = (PASS == 0 ? A.p1 : A.p2) + g * k;
    cluster_dots<kClu>(C, 0, k, rank, kClu, [&](int j, double2 h) { out[j] = h; });
    cluster_barrier();  // no CTA exits while others read its shared memory
    return;
  }
  if (t == 0) C.npart = block_nrm(C.S, col_warps(k));  // a row group's first warp has its rows
  cluster_barrier();
  if (rank == 0 && t < 32) {
    double s = t < kClu ? cluster_load(&C.npart, t) : 0.0;
    s = warp_sum(s);
    unsigned last = 0;
    if (t == 0) {
      A.np[g] = s;
      __threadfence();
      last = atomicAdd(A.counter, 1u) == (unsigned)A.G - 1;
    }
    if (__shfl_sync(0xffffffffu, last, 0)) {  // the last cluster adds the norms up
      __threadfence();
      double q = t < A.G ? __ldcg(A.np + t) : 0.0;
      q = sqrt(warp_sum(q));
      if (t == 0) {
        *A.d_norm = q;
        *A.counter = 0u;
      }
    }
  }
  cluster_barrier();
}

// launch configuration of a cluster kernel (cfg keeps a pointer to attr); chained: see launch_chained
inline void cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&attr)[2], int ctas, unsigned clusters,
                           cudaStream_t st, bool chained) {
  cfg = cudaLaunchConfig_t{};
  cfg.gridDim = dim3(clusters * ctas);
  cfg.blockDim = dim3(kColThreads);
  cfg.stream = st;
  attr[0] = cudaLaunchAttribute{};
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = ctas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1] = cudaLaunchAttribute{};
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chained ? 2 : 1;
}

}  // namespace gs

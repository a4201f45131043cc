// Matrix-vector products of the compressed matrix (Section 4, Eqs. mvm1-mvm3,
// figure "Fast forward and backward transformation"): y = G~ x and the adjoint
// y = G~^* x, for one or several right-hand sides.
//
// The products read every stored entry once, so the nearfield blocks (most of
// the representation) set their time: HBM in FP32, the narrow FP64 pipe in
// FP64 (4 fused multiply-adds per entry and right-hand side).
//
// Right-hand sides are taken NR at a time from one read of the matrix; a
// chunk's unused slots (nr < NR) repeat slot 0 and are not written.
#include <algorithm>

#include "dh2_check.cuh"
#include "dh2_internal.h"
#include "dh2_ops.cuh"

namespace dh2 {

namespace {

template <typename T>
__device__ __forceinline__ C2<T> czero() { return C2<T>{T(0), T(0)}; }
// acc + a b and acc + conj(a) b as fused multiply-adds
template <typename T>
__device__ __forceinline__ C2<T> cfma(C2<T> acc, C2<T> a, C2<T> b) {
  acc.re = fma(a.re, b.re, acc.re);
  acc.im = fma(a.re, b.im, acc.im);
  acc.re = fma(-a.im, b.im, acc.re);
  acc.im = fma(a.im, b.re, acc.im);
  return acc;
}
template <typename T>
__device__ __forceinline__ C2<T> cfma_conj(C2<T> acc, C2<T> a, C2<T> b) {
  acc.re = fma(a.re, b.re, acc.re);
  acc.im = fma(a.re, b.im, acc.im);
  acc.re = fma(a.im, b.im, acc.re);
  acc.im = fma(-a.im, b.re, acc.im);
  return acc;
}
// one vector reduction in FP32, two scalar ones in FP64
__device__ __forceinline__ void red_add(C2<float>* p, C2<float> v) {
  atomicAdd(reinterpret_cast<float2*>(p), make_float2(v.re, v.im));
}
__device__ __forceinline__ void red_add(C2<double>* p, C2<double> v) {
  atomicAdd(&p->re, v.re);
  atomicAdd(&p->im, v.im);
}
__device__ __forceinline__ C2<float> ldg(const C2<float>* p) {
  const float2 v = __ldg(reinterpret_cast<const float2*>(p));
  return C2<float>{v.x, v.y};
}
__device__ __forceinline__ C2<double> ldg(const C2<double>* p) {
  const double2 v = __ldg(reinterpret_cast<const double2*>(p));
  return C2<double>{v.x, v.y};
}

// Sums of 8 values per lane over a warp in 9 shuffles (each exchange halves
// the values a lane holds): the sum of v[i] ends in the lanes with
// col_of(lane) == i.
__device__ __forceinline__ int col_of(int lane) {
  return ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
}
template <typename T>
__device__ __forceinline__ T sum8(const T (&v)[8], int lane) {
  const bool b4 = (lane >> 4) & 1, b3 = (lane >> 3) & 1, b2 = (lane >> 2) & 1;
  T w4[4], w2[2];
#pragma unroll
  for (int i = 0; i < 4; ++i)
    w4[i] = (b4 ? v[4 + i] : v[i]) + __shfl_xor_sync(0xffffffffu, b4 ? v[i] : v[4 + i], 16);
#pragma unroll
  for (int i = 0; i < 2; ++i)
    w2[i] = (b3 ? w4[2 + i] : w4[i]) + __shfl_xor_sync(0xffffffffu, b3 ? w4[i] : w4[2 + i], 8);
  T w1 = (b2 ? w2[1] : w2[0]) + __shfl_xor_sync(0xffffffffu, b2 ? w2[0] : w2[1], 4);
  w1 += __shfl_xor_sync(0xffffffffu, w1, 2);
  w1 += __shfl_xor_sync(0xffffffffu, w1, 1);
  return w1;
}

// Right-hand side slots of a chunk: offsets rh * stride, unused ones at slot 0.
template <int NR>
struct Rhs {
  int64_t o[NR];
  __device__ __forceinline__ Rhs(int rh0, int nr, int64_t stride) {
#pragma unroll
    for (int k = 0; k < NR; ++k) o[k] = (int64_t)(rh0 + (k < nr ? k : 0)) * stride;
  }
};

// A launch takes right-hand sides [first, first + count), NR per blockIdx.y: the
// first of this CTA's, and how many it has.
template <int NR>
__device__ __forceinline__ int chunk_begin(int rh0) { return rh0 + blockIdx.y * NR; }
template <int NR>
__device__ __forceinline__ int chunk_width(int count) { return min(NR, count - (int)blockIdx.y * NR); }

// ---------------------------------------------------------------- nearfield
// y|_t += G_b x|_s over the inadmissible blocks (ADJ: y|_s += G_b^* x|_t), a
// unit (a slab of one row cluster's rows, or of one column cluster's columns,
// and a run of its blocks) per CTA.  The blocks pass through a ring of
// shared-memory stages filled by cp.async, in pieces of at most kNearElems
// entries with their part of the vectors.  A thread keeps one row (column) i =
// tid % mr of the unit and every (128 / mr)-th entry of it, and the sums of all
// the unit's blocks stay in registers until one reduction and one atomic
// addition per row.  Product: a piece is a run of columns, contiguous in the
// nearfield copy (16-byte copies), and consecutive threads read consecutive
// entries.  Adjoint: a piece is a run of rows, its columns staged at an odd
// distance so that threads on consecutive columns read without bank conflicts.
// FP32 is bound by HBM: two stages ahead in 4 CTAs per SM keep ~100 KB per SM in
// flight; n = 32768, one vector: 975 us, 6.4 TB/s (a row per thread with loads
// from global memory: 1808 us; eight loads in flight per thread: 2245 us, each
// round of a 40-row block paid a DRAM and then an L2 latency).  FP64 is bound by
// its pipe, 4 fused multiply-adds per entry and vector: n = 8192, eight
// vectors: 3.0 ms against 4.4 ms with 6 operations.
template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

template <typename T, int NR>
__device__ __forceinline__ void leaf_unit(const MvArgs<T>& a, const int32_t* __restrict__ pairs, const NearUnit& u,
                                          int rh0, int nr, int nrhs, C2<T>* __restrict__ y, int64_t n, C2<T>* red);
template <typename T, int NR, bool ADJ>
__global__ void __launch_bounds__(128) mv_near(MvArgs<T> a, int first, int count, const C2<T>* __restrict__ x,
                                               C2<T>* __restrict__ y, int64_t n, const int32_t* __restrict__ pairs,
                                               const NearUnit* __restrict__ leafs, int nrhs) {
  const int rh0 = chunk_begin<NR>(first), nr = chunk_width<NR>(count);
  // stages (static shared memory, below 48 KB); FP64 takes half a piece at a time
  constexpr int S = NR <= 4 ? 3 : 2;
  constexpr int SG = kNearElems * 4 / (int)sizeof(T), SX = kNearPiece * NR * 4 / (int)sizeof(T);
  __shared__ __align__(16) C2<T> sm[S * (SG + SX)];
  __shared__ int sw[S];  // width of the piece in each stage, 0 past the last
  static_assert(128 * NR <= S * (SG + SX), "the reduction reuses the stages");
  if ((int)blockIdx.x >= a.nunits) {  // a small product's leaf step in the same launch
    leaf_unit<T, NR>(a, pairs, leafs[blockIdx.x - a.nunits], rh0, nr, nrhs, y, n, sm);
    return;
  }
  const NearUnit u = a.units[blockIdx.x];
  const int tid = threadIdx.x;
  const int mr = u.cw, r = tid % mr, c = tid / mr, cg = 128 / mr;
  const NearItem* items = a.items + u.first;
  // the piece to copy next: item qi (it; the one after it in nx), from entry qj
  int qi = 0, qj = 0;
  NearItem it = items[0], nx = items[u.count > 1 ? 1 : 0];
  // copies of that piece and of its part of the vectors into stage s
  auto issue = [&](int s) {
    if (qi >= u.count) {
      if (tid == 0) sw[s] = 0;
      return;
    }
    C2<T>* g = sm + s * (SG + SX);
    const int w = min(sizeof(T) == 4 ? it.pw : (it.pw >> 1), it.w - qj);
    if (tid == 0) sw[s] = w;
    const int cnt = w * mr;
    const int64_t ld = a.near ? it.ld : a.ld;
    if constexpr (ADJ) {
      const C2<T>* src = a.near ? a.near + it.off + qj + u.c0 * ld : a.G + (it.o0 + qj) + u.out * ld;
      const int lw = w | 1, di = 128 % w, dj = 128 / w;
      for (int i = tid % w, j = tid / w; j < mr;) {
        cp_async<sizeof(C2<T>)>(g + j * lw + i, src + i + j * ld);
        i += di;
        j += dj;
        if (i >= w) {
          i -= w;
          ++j;
        }
      }
    } else if (a.near && it.ld == mr) {
      const C2<T>* src = a.near + it.off + qj * mr;
      if constexpr (sizeof(T) == 4) {  // an odd count copies the padding entry too
        for (int e = 2 * tid; e < cnt; e += 256) cp_async<16>(g + e, src + e);
      } else {
        for (int e = tid; e < cnt; e += 128) cp_async<16>(g + e, src + e);
      }
    } else {  // a slab of taller blocks, or the blocks in place in G
      const C2<T>* src = a.near ? a.near + it.off + u.c0 + qj * ld : a.G + (it.o0 + qj) * ld + u.out;
      for (int e = tid; e < cnt; e += 128) cp_async<sizeof(C2<T>)>(g + e, src + e % mr + (e / mr) * ld);
    }
    C2<T>* xs = g + SG;
    const C2<T>* xg = x + it.o0 + qj;
    if constexpr (NR == 1) {
      if (tid < w) cp_async<sizeof(C2<T>)>(xs + tid, xg + tid + rh0 * n);
    } else {
      for (int e = tid; e < w * nr; e += 128) {
        const int k = e / w, j = e - k * w;
        cp_async<sizeof(C2<T>)>(xs + j * NR + k, xg + j + (rh0 + k) * n);
      }
    }
    qj += w;
    if (qj >= it.w) {
      qj = 0;
      ++qi;
      it = nx;
      if (qi + 1 < u.count) nx = items[qi + 1];
    }
  };
  // sums in two steps: of a piece (where the additions cost pipe time, of several:
  // 5 to 8 vectors in FP32 two, forward 5% slower by single ones; FP64 eight half
  // pieces), and of those.  One chain over the unit's ~1600 columns had
  // 1.2 to 1.7 times the rounding error of block after block (n = 8192, leaf 64,
  // against FP64: 4.7e-7, by block 2.7e-7, now 1.5e-7), for 1% of the time in
  // FP32 (n = 32768, one vector: 1162 -> 1171 us) and 2% in FP64.  FP64, one and
  // two vectors: four chains instead, which as well are a quarter as long (the
  // second sums had cost 8%)
  constexpr int U = sizeof(T) == 8 && NR <= 2 ? 4 : 1;
  constexpr int FOLD = sizeof(T) == 8 ? 8 : NR < 8 || ADJ ? 1 : 2;
  C2<T> acc[U][NR], sum[NR];
#pragma unroll
  for (int k = 0; k < NR; ++k) {
    sum[k] = czero<T>();
#pragma unroll
    for (int u = 0; u < U; ++u) acc[u][k] = czero<T>();
  }
  auto fold = [&]() {
#pragma unroll
    for (int k = 0; k < NR; ++k)
#pragma unroll
      for (int u = 0; u < U; ++u) {
        sum[k].re += acc[u][k].re;
        sum[k].im += acc[u][k].im;
        acc[u][k] = czero<T>();
      }
  };
#pragma unroll
  for (int s = 0; s < S - 1; ++s) {
    issue(s);
    cp_async_commit();
  }
  for (int q = 0;; ++q) {
    cp_async_wait<S - 2>();
    __syncthreads();  // piece q has landed; the stage of piece q - 1 is free
    const int w = sw[q % S];
    if (w == 0) break;
    issue((q + S - 1) % S);
    cp_async_commit();
    const C2<T>* g = sm + (q % S) * (SG + SX) + (ADJ ? r * (w | 1) : r);
    const C2<T>* xs = sm + (q % S) * (SG + SX) + SG;
    if (c < cg) {
      auto add = [&](int j, int u) {
        const C2<T> v = ADJ ? g[j] : g[j * mr];
#pragma unroll
        for (int k = 0; k < NR; ++k)
          acc[u][k] = ADJ ? cfma_conj(acc[u][k], v, xs[j * NR + k]) : cfma(acc[u][k], v, xs[j * NR + k]);
      };
      if constexpr (U == 1) {
#pragma unroll 4
        for (int j = c; j < w; j += cg) add(j, 0);
      } else {
        int j = c;
        for (; j + (U - 1) * cg < w; j += U * cg)
#pragma unroll
          for (int u = 0; u < U; ++u) add(j + u * cg, u);
        for (; j < w; j += cg) add(j, 0);
        // the chain that took the rest goes to the back
#pragma unroll
        for (int k = 0; k < NR; ++k) {
          const C2<T> t = acc[0][k];
#pragma unroll
          for (int u = 0; u + 1 < U; ++u) acc[u][k] = acc[u + 1][k];
          acc[U - 1][k] = t;
        }
      }
    }
    if (U == 1 && q % FOLD == FOLD - 1) fold();
  }
  fold();
  // (no copy is in flight: past the last piece nothing was issued)
  __syncthreads();
  C2<T>* red = sm;
#pragma unroll
  for (int k = 0; k < NR; ++k) red[k * 128 + tid] = sum[k];
  __syncthreads();
  for (int e = tid; e < mr * nr; e += 128) {
    const int i = e % mr, k = e / mr;
    C2<T> s = red[k * 128 + i];
    for (int cc = 1; cc < cg; ++cc) {
      s.re += red[k * 128 + cc * mr + i].re;
      s.im += red[k * 128 + cc * mr + i].im;
    }
    red_add(y + u.out + i + (int64_t)(rh0 + k) * n, s);
  }
}

// ---------------------------------------------------------------- transformations
// out_q = sum_i conj(M(i, q)) v_i for the columns q0 .. q0 + 7 of a p x k
// matrix (column-major, ld), by one warp; get(i, o) is entry i of a vector.
template <typename T, int NR, typename Get>
__device__ __forceinline__ void cols_dot(const C2<T>* M, int ld, int p, int k, int q0, int lane, const Get& get,
                                         C2<T> (&out)[NR]) {
  T vr[NR][8], vi[NR][8];
#pragma unroll
  for (int h = 0; h < NR; ++h)
#pragma unroll
    for (int i = 0; i < 8; ++i) vr[h][i] = vi[h][i] = T(0);
  for (int r = lane; r < p; r += 32) {
    C2<T> m[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) m[i] = q0 + i < k ? ldg(M + r + (int64_t)(q0 + i) * ld) : czero<T>();
#pragma unroll
    for (int h = 0; h < NR; ++h) {
      const C2<T> v = get(r, h);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const C2<T> s = cfma_conj(C2<T>{vr[h][i], vi[h][i]}, m[i], v);
        vr[h][i] = s.re;
        vi[h][i] = s.im;
      }
    }
  }
#pragma unroll
  for (int h = 0; h < NR; ++h) out[h] = C2<T>{sum8(vr[h], lane), sum8(vi[h], lane)};
}

// forward transformation, leaves: xh_sc = W_sc^* x|_s (Eq. mvm1), one warp per
// pair; y0 (nzero entries, or NULL): a small product's result, zeroed on the way
template <typename T, int NR>
__global__ void __launch_bounds__(128) mv_forward_leaf(SideView<T> W, const int32_t* __restrict__ pairs, int np,
                                                       int first, int count, const C2<T>* __restrict__ x, int nrhs,
                                                       int64_t n, C2<T>* __restrict__ xh,
                                                       const int64_t* __restrict__ hoff, C2<T>* __restrict__ y0,
                                                       int64_t nzero) {
  const int rh0 = chunk_begin<NR>(first), nr = chunk_width<NR>(count);
  if (y0 && blockIdx.y == 0)
    for (int64_t i = blockIdx.x * (int64_t)128 + threadIdx.x; i < nzero; i += (int64_t)gridDim.x * 128)
      y0[i] = czero<T>();
  const int w = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (w >= np) return;
  const int pid = pairs[w];
  const int k = W.rank[pid];
  const int cl = W.cluster[pid];
  const int m = W.csize[cl];
  const C2<T>* xs = x + W.cstart[cl];
  const C2<T>* Q = W.Q + W.Qoff[pid];
  const Rhs<NR> rh(rh0, nr, n);
  C2<T>* o = xh + hoff[pid] * nrhs + (int64_t)rh0 * k;
  const int col = col_of(lane);
  for (int q0 = 0; q0 < k; q0 += 8) {
    C2<T> s[NR];
    cols_dot<T, NR>(Q, m, m, k, q0, lane, [&](int r, int h) { return ldg(xs + r + rh.o[h]); }, s);
#pragma unroll
    for (int h = 0; h < NR; ++h)
      if ((lane & 3) == 0 && q0 + col < k && h < nr) o[q0 + col + (int64_t)h * k] = s[h];
  }
}

// forward transformation, non-leaves: xh_sc = [E_s1c; E_s2c]^* [xh_s1c'; xh_s2c'],
// one CTA per pair, its warps take 8 columns each
template <typename T, int NR>
__global__ void __launch_bounds__(128) mv_forward_up(SideView<T> W, const int32_t* __restrict__ pairs, int first, int count,
                                                     int nrhs, C2<T>* xh, const int64_t* __restrict__ hoff) {
  const int rh0 = chunk_begin<NR>(first), nr = chunk_width<NR>(count);
  const int pid = pairs[blockIdx.x];
  const int lane = threadIdx.x & 31;
  const int k = W.rank[pid];
  const int s0 = W.son[2 * pid], s1 = W.son[2 * pid + 1];
  const int k0 = W.rank[s0], k1 = W.rank[s1];
  const C2<T>* E = W.Q + W.Qoff[pid];
  const C2<T>* x0 = xh + hoff[s0] * nrhs;
  const C2<T>* x1 = xh + hoff[s1] * nrhs;
  C2<T>* o = xh + hoff[pid] * nrhs + (int64_t)rh0 * k;
  const int col = col_of(lane);
  for (int q0 = 8 * (threadIdx.x >> 5); q0 < k; q0 += 32) {
    C2<T> s[NR];
    cols_dot<T, NR>(E, W.rowcap[pid], k0 + k1, k, q0, lane,
                    [&](int r, int h) {
                      const int64_t v = rh0 + (h < nr ? h : 0);
                      return r < k0 ? x0[r + v * k0] : x1[r - k0 + v * k1];
                    },
                    s);
#pragma unroll
    for (int h = 0; h < NR; ++h)
      if ((lane & 3) == 0 && q0 + col < k && h < nr) o[q0 + col + (int64_t)h * k] = s[h];
  }
}

// A pair's blocks as a warp walks them (blocks first, first + step, ...): the
// list entry of a later block, and the other pair's rank and coefficient offset
// of the next one, are loaded while a block's products run, so a block costs
// one load latency instead of a chain of four.
struct OwnWalk {
  const OwnItem* own;
  const int32_t* rank;
  const int64_t* hoff;
  int64_t e, e1;
  int step;
  OwnItem cur, nxt;
  int k, kn;
  int64_t ho, hon;
  __device__ __forceinline__ OwnWalk(const OwnItem* own_, const int32_t* rank_, const int64_t* hoff_, int64_t e0,
                                     int64_t e1_, int step_)
      : own(own_), rank(rank_), hoff(hoff_), e(e0), e1(e1_), step(step_) {
    cur = nxt = OwnItem{0, 0, 0};
    k = kn = 0;
    ho = hon = 0;
    if (e < e1) cur = own[e];
    if (e + step < e1) nxt = own[e + step];
    if (e < e1) {
      k = rank[cur.pair];
      ho = hoff[cur.pair];
    }
  }
  __device__ __forceinline__ bool live() const { return e < e1; }
  __device__ __forceinline__ void prefetch() {  // before the products of the current block
    if (e + step < e1) {
      kn = rank[nxt.pair];
      hon = hoff[nxt.pair];
    }
  }
  __device__ __forceinline__ void next() {
    e += step;
    cur = nxt;
    k = kn;
    ho = hon;
    if (e + step < e1) nxt = own[e + step];
  }
};

// coupling: yh_tc = sum over own blocks b of S_b xh_sc (Eq. mvm2), one CTA per
// pair, the blocks dealt to its warps; in a warp a lane keeps row r = lane % kr
// (at most 32 rows a pass) and every (32 / kr)-th column, so S_b is read in
// order and the sums of all blocks stay in registers until one reduction.
// Bound by the latency of a block's few loads (a pair has 8 blocks on average;
// one warp per pair took 185 us at n = 32768, four 138).
template <typename T, int NR>
__global__ void __launch_bounds__(128) mv_coupling(MvArgs<T> a, int first, int count, int nrhs) {
  const int rh0 = chunk_begin<NR>(first), nr = chunk_width<NR>(count);
  __shared__ C2<T> red[4][32 * NR];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int pid = blockIdx.x;
  const int kt = a.V.rank[pid];
  const int64_t e0 = a.own_ptr[pid], e1 = a.own_ptr[pid + 1];
  for (int r0 = 0; r0 < kt; r0 += 32) {
    const int kr = min(32, kt - r0);
    const int r = lane % kr, c = lane / kr, cg = 32 / kr;
    C2<T> acc[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) acc[k] = czero<T>();
    for (OwnWalk b(a.own, a.W.rank, a.xhoff, e0 + warp, e1, 4); b.live(); b.next()) {
      b.prefetch();
      const C2<T>* S = a.S + b.cur.soff + r0 + r;
      const C2<T>* xs = a.xh + b.ho * nrhs;
      const Rhs<NR> rh(rh0, nr, b.k);
      if (c < cg)
#pragma unroll 4
        for (int l = c; l < b.k; l += cg) {
          const C2<T> s = ldg(S + l * kt);
#pragma unroll
          for (int k = 0; k < NR; ++k) acc[k] = cfma(acc[k], s, ldg(xs + l + rh.o[k]));
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NR; ++k) red[warp][k * 32 + lane] = acc[k];
    __syncthreads();
    for (int e = threadIdx.x; e < kr * nr; e += 128) {
      const int i = e % kr, k = e / kr;
      C2<T> s = czero<T>();
      for (int g = 0; g < 4; ++g)
        for (int cc = 0; cc < cg; ++cc) {
          s.re += red[g][k * 32 + cc * kr + i].re;
          s.im += red[g][k * 32 + cc * kr + i].im;
        }
      a.yh[a.yhoff[pid] * nrhs + r0 + i + (int64_t)(rh0 + k) * kt] = s;
    }
  }
}

// adjoint coupling: yh_sc = sum over the column pair's blocks b of S_b^* xh_tc;
// in a warp two lanes per column of S_b and 16 columns per pass
template <typename T, int NR>
__global__ void __launch_bounds__(128) mv_coupling_adj(MvArgs<T> a, int first, int count, int nrhs) {
  const int rh0 = chunk_begin<NR>(first), nr = chunk_width<NR>(count);
  __shared__ C2<T> red[4][16 * NR];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int pid = blockIdx.x;
  const int kout = a.V.rank[pid];  // rank of this column pair
  const int64_t e0 = a.own_ptr[pid], e1 = a.own_ptr[pid + 1];
  for (int q0 = 0; q0 < kout; q0 += 16) {
    const int qq = q0 + (lane >> 1);
    C2<T> acc[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) acc[k] = czero<T>();
    for (OwnWalk b(a.own, a.W.rank, a.xhoff, e0 + warp, e1, 4); b.live(); b.next()) {
      b.prefetch();
      const int kin = b.k;  // rank of the block's row pair; S_b is kin x kout
      const C2<T>* S = a.S + b.cur.soff + (int64_t)qq * kin;
      const C2<T>* xs = a.xh + b.ho * nrhs;
      const Rhs<NR> rh(rh0, nr, kin);
      if (qq < kout)
#pragma unroll 4
        for (int l = lane & 1; l < kin; l += 2) {
          const C2<T> s = ldg(S + l);
#pragma unroll
          for (int k = 0; k < NR; ++k) acc[k] = cfma_conj(acc[k], s, ldg(xs + l + rh.o[k]));
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      acc[k].re += __shfl_xor_sync(0xffffffffu, acc[k].re, 1);
      acc[k].im += __shfl_xor_sync(0xffffffffu, acc[k].im, 1);
      if (!(lane & 1)) red[warp][k * 16 + (lane >> 1)] = acc[k];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 16 * nr; e += 128) {
      const int i = e & 15, k = e >> 4;
      if (q0 + i < kout) {
        C2<T> s = czero<T>();
        for (int g = 0; g < 4; ++g) {
          s.re += red[g][e].re;
          s.im += red[g][e].im;
        }
        a.yh[a.yhoff[pid] * nrhs + q0 + i + (int64_t)(rh0 + k) * kout] = s;
      }
    }
  }
}

// backward transformation: yh_t'c' += E_t'c yh_tc over the father pairs (t, c)
// with sd(c) = c', gathered per son pair (figure "Fast forward and backward
// transformation", right); one warp per pair, rows and columns dealt to its
// lanes as in the coupling (above 32 rows a lane takes every 32nd row)
template <typename T, int NR>
__global__ void __launch_bounds__(128) mv_backward_down(MvArgs<T> a, const int32_t* __restrict__ pairs, int np,
                                                        int first, int count, int nrhs) {
  const int rh0 = chunk_begin<NR>(first), nr = chunk_width<NR>(count);
  __shared__ C2<T> red[4][32 * NR];
  const int wl = threadIdx.x >> 5, w = blockIdx.x * 4 + wl, lane = threadIdx.x & 31;
  if (w >= np) return;
  const int pid = pairs[w];
  const int k = a.V.rank[pid];
  const int64_t f0 = a.par_ptr[pid], f1 = a.par_ptr[pid + 1];
  if (k == 0 || f0 == f1) return;
  C2<T>* yo = a.yh + a.yhoff[pid] * nrhs + (int64_t)rh0 * k;
  for (int r0 = 0; r0 < k; r0 += 32) {
    const int kr = min(32, k - r0);
    const int r = lane % kr, c = lane / kr, cg = 32 / kr;
    C2<T> acc[NR];
#pragma unroll
    for (int h = 0; h < NR; ++h) acc[h] = czero<T>();
    if (c < cg)
      for (int64_t e = f0; e < f1; ++e) {
        const int fp = a.par_pair[e];
        const int kf = a.V.rank[fp];
        const int ldq = a.V.rowcap[fp];
        const int eoff = a.par_son[e] == 0 ? 0 : a.V.rank[a.V.son[2 * fp]];
        const C2<T>* E = a.V.Q + a.V.Qoff[fp] + eoff + r0 + r;
        const C2<T>* yf = a.yh + a.yhoff[fp] * nrhs;
        const Rhs<NR> rh(rh0, nr, kf);
#pragma unroll 4
        for (int l = c; l < kf; l += cg) {
          const C2<T> v = ldg(E + (int64_t)l * ldq);
#pragma unroll
          for (int h = 0; h < NR; ++h) acc[h] = cfma(acc[h], v, yf[l + rh.o[h]]);
        }
      }
    __syncwarp();
#pragma unroll
    for (int h = 0; h < NR; ++h) red[wl][h * 32 + lane] = acc[h];
    __syncwarp();
    for (int e = lane; e < kr * nr; e += 32) {
      const int i = e % kr, h = e / kr;
      C2<T> s = yo[r0 + i + (int64_t)h * k];
      for (int cc = 0; cc < cg; ++cc) {
        s.re += red[wl][h * 32 + cc * kr + i].re;
        s.im += red[wl][h * 32 + cc * kr + i].im;
      }
      yo[r0 + i + (int64_t)h * k] = s;
    }
  }
}

// leaves: y|_t += V_tc yh_tc (Eq. mvm3), one CTA per run of pairs of one leaf
// cluster (unit: pairs first .. first + count - 1 of the list, rows as in
// mv_near), one atomic addition per row and run
template <typename T, int NR>
__device__ __forceinline__ void leaf_unit(const MvArgs<T>& a, const int32_t* __restrict__ pairs, const NearUnit& u,
                                          int rh0, int nr, int nrhs, C2<T>* __restrict__ y, int64_t n, C2<T>* red) {
  const int tid = threadIdx.x;
  const int m = u.cw, r = tid % m, c = tid / m, cg = 128 / m;
  C2<T> acc[NR];
#pragma unroll
  for (int h = 0; h < NR; ++h) acc[h] = czero<T>();
  if (c < cg)
    for (int q = 0; q < u.count; ++q) {
      const int pid = pairs[u.first + q];
      const int k = a.V.rank[pid];
      const C2<T>* Q = a.V.Q + a.V.Qoff[pid] + r;
      const C2<T>* yh = a.yh + a.yhoff[pid] * nrhs;
      const Rhs<NR> rh(rh0, nr, k);
#pragma unroll 4
      for (int l = c; l < k; l += cg) {
        const C2<T> v = ldg(Q + l * m);
#pragma unroll
        for (int h = 0; h < NR; ++h) acc[h] = cfma(acc[h], v, ldg(yh + l + rh.o[h]));
      }
    }
#pragma unroll
  for (int h = 0; h < NR; ++h) red[h * 128 + tid] = acc[h];
  __syncthreads();
  for (int e = tid; e < m * nr; e += 128) {
    const int i = e % m, h = e / m;
    C2<T> s = red[h * 128 + i];
    for (int cc = 1; cc < cg; ++cc) {
      s.re += red[h * 128 + cc * m + i].re;
      s.im += red[h * 128 + cc * m + i].im;
    }
    red_add(y + u.out + i + (int64_t)(rh0 + h) * n, s);
  }
}
template <typename T, int NR>
__global__ void __launch_bounds__(128) mv_backward_leaf(MvArgs<T> a, const int32_t* __restrict__ pairs,
                                                        const NearUnit* __restrict__ units, int first, int count,
                                                        int nrhs, C2<T>* __restrict__ y, int64_t n) {
  const int rh0 = chunk_begin<NR>(first), nr = chunk_width<NR>(count);
  __shared__ C2<T> red[128 * NR];
  leaf_unit<T, NR>(a, pairs, units[blockIdx.x], rh0, nr, nrhs, y, n, red);
}

// The right-hand sides in chunks of a compiled width, those of one width in one
// launch: f(width constant, first, count), chunk blockIdx.y of the launch's
// columns [first, first + count).  (One launch per chunk took n = 2000, sixteen
// vectors, 146 us; every vector in one launch of the old kernels 126.)  MOST: the
// widest kernel that keeps its sums in registers.  FP32
// rounds 5 to 7 up to 8 (one read of the matrix; the extra multiply-adds cost
// less than a second read); FP64 takes exact widths (they would cost the narrow
// FP64 pipe).
template <int NR>
dim3 chunk_grid(int x, int count) { return dim3((unsigned)x, (unsigned)((count + NR - 1) / NR)); }
template <int V>
struct Int {
  static constexpr int value = V;
};
constexpr int kMaxChunks = 65535;  // a grid's y extent
template <typename T, int MOST, typename F>
void rhs_chunks(int nrhs, const F& f, int most = MOST) {
  constexpr int UP = sizeof(T) == 4 ? 3 : 0;  // columns a chunk of 8 may lack
  for (int rh = 0; rh < nrhs;) {
    const int left = nrhs - rh;
    int nr;
    if (MOST >= 8 && most >= 8 && left >= 8 - UP) {
      const int64_t full = (left + (int64_t)UP) / 8;
      nr = (int)std::min<int64_t>(left, 8 * std::min<int64_t>(full, kMaxChunks));
      f(Int<(MOST >= 8 ? 8 : 1)>{}, rh, nr);
    } else if (MOST >= 4 && most >= 4 && left >= 4) {
      nr = 4 * std::min(left / 4, kMaxChunks);
      f(Int<(MOST >= 4 ? 4 : 1)>{}, rh, nr);
    } else if (MOST >= 4 && most >= 4 && left == 3) {
      nr = 3;
      f(Int<(MOST >= 4 ? 3 : 1)>{}, rh, nr);
    } else if (most >= 2 && left >= 2) {
      nr = 2 * std::min(left / 2, kMaxChunks);
      f(Int<2>{}, rh, nr);
    } else {
      nr = std::min(left, kMaxChunks);
      f(Int<1>{}, rh, nr);
    }
    rh += nr;
  }
}
// ---------------------------------------------------------------- lists
// items: one thread per inadmissible block, at the next free place of its
// cluster (a cluster's blocks are summed, so their order is free)
__global__ void __launch_bounds__(256) near_items_kernel(NearFill f) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= f.nblocks) return;
  const int b = f.blocks[i];
  const int c = f.own[b], o = f.other[b];
  const int w = f.csize[o];
  // the adjoint's stages hold the columns at an odd distance, w | 1: the widest
  // piece is twice an odd number, so that this fits its FP64 half as well
  const int fit = min(kNearPiece, kNearElems / near_slab(f.csize[c]) - f.sd);
  const int most = f.sd ? ((fit - 2) & ~3) + 2 : fit & ~1;
  const int np = (w + most - 1) / most;
  f.items[f.item_begin[c] + atomicAdd(f.cursor + c, 1)] =
      NearItem{f.near_off[b], f.cstart[o], w, f.csize[f.bt[b]], min(most, ((w + np - 1) / np + 1) & ~1)};
}
// units: one warp per cluster, its items in runs of equal length
__global__ void __launch_bounds__(256) near_units_kernel(NearFill f) {
  const int c = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (c >= f.nclusters) return;
  const int i0 = f.item_begin[c], ni = f.item_begin[c + 1] - i0;
  const int u0 = f.unit_begin[c], nu = f.unit_begin[c + 1] - u0;
  if (nu == 0) return;
  const int mine = f.csize[c], slabs = near_slabs(mine), slab = near_slab(mine);
  const int runs = nu / slabs, per = (ni + runs - 1) / runs;
  for (int u = threadIdx.x & 31; u < nu; u += 32) {
    const int run = u / slabs, c0 = (u % slabs) * slab;
    f.units[u0 + u] = NearUnit{i0 + run * per, min(per, ni - run * per), c0, min(slab, mine - c0), f.cstart[c] + c0, 0};
  }
}
__global__ void __launch_bounds__(256) own_items_kernel(const int32_t* __restrict__ blk, int64_t n,
                                                        const int64_t* __restrict__ Soff,
                                                        const int32_t* __restrict__ other_pair,
                                                        OwnItem* __restrict__ own) {
  const int64_t i = blockIdx.x * (int64_t)256 + threadIdx.x;
  if (i < n) own[i] = OwnItem{Soff[blk[i]], other_pair[blk[i]], 0};
}

}  // namespace

void launch_mv_lists(const NearFill& f, const int32_t* own_blk, int64_t nown, const int64_t* Soff,
                     const int32_t* other_pair, OwnItem* own, cudaStream_t st) {
  if (f.nblocks > 0) {
    near_items_kernel<<<(f.nblocks + 255) / 256, 256, 0, st>>>(f);
    near_units_kernel<<<(f.nclusters + 7) / 8, 256, 0, st>>>(f);
  }
  if (nown > 0) own_items_kernel<<<(unsigned)((nown + 255) / 256), 256, 0, st>>>(own_blk, nown, Soff, other_pair, own);
}

template <typename T>
void launch_mv_forward_leaf(const SideView<T>& W, const int32_t* pairs, int np, const C2<T>* x, int nrhs, int64_t n,
                            C2<T>* xh, const int64_t* hoff, C2<T>* y0, cudaStream_t st) {
  if (np <= 0) return;
  rhs_chunks<T, sizeof(T) == 4 ? 4 : 2>(nrhs, [&](auto w, int rh, int nr) {
    mv_forward_leaf<T, decltype(w)::value>
        <<<chunk_grid<decltype(w)::value>((np + 3) / 4, nr), 128, 0, st>>>(W, pairs, np, rh, nr, x, nrhs, n, xh, hoff,
                                                                          rh == 0 ? y0 : nullptr, n * nrhs);
  });
}
template <typename T>
void launch_mv_forward_up(const SideView<T>& W, const int32_t* pairs, int np, int nrhs, C2<T>* xh,
                          const int64_t* hoff, cudaStream_t st) {
  if (np <= 0) return;
  rhs_chunks<T, sizeof(T) == 4 ? 4 : 2>(nrhs, [&](auto w, int rh, int nr) {
    mv_forward_up<T, decltype(w)::value>
        <<<chunk_grid<decltype(w)::value>(np, nr), 128, 0, st>>>(W, pairs, rh, nr, nrhs, xh, hoff);
  });
}
template <typename T>
void launch_mv_coupling(const MvArgs<T>& a, int npairs_row, int nrhs, cudaStream_t st) {
  if (npairs_row <= 0) return;
  rhs_chunks<T, 8>(nrhs, [&](auto w, int rh, int nr) {
    mv_coupling<T, decltype(w)::value><<<chunk_grid<decltype(w)::value>(npairs_row, nr), 128, 0, st>>>(a, rh, nr, nrhs);
  });
}
template <typename T>
void launch_mv_coupling_adj(const MvArgs<T>& a, int npairs_col, int nrhs, cudaStream_t st) {
  if (npairs_col <= 0) return;
  rhs_chunks<T, 8>(nrhs, [&](auto w, int rh, int nr) {
    mv_coupling_adj<T, decltype(w)::value><<<chunk_grid<decltype(w)::value>(npairs_col, nr), 128, 0, st>>>(a, rh, nr, nrhs);
  });
}
template <typename T>
void launch_mv_backward_down(const MvArgs<T>& a, const int32_t* pairs, int np, int nrhs, cudaStream_t st) {
  if (np <= 0) return;
  rhs_chunks<T, 8>(nrhs, [&](auto w, int rh, int nr) {
    mv_backward_down<T, decltype(w)::value>
        <<<chunk_grid<decltype(w)::value>((np + 3) / 4, nr), 128, 0, st>>>(a, pairs, np, rh, nr, nrhs);
  });
}
template <typename T>
void launch_mv_backward_leaf(const MvArgs<T>& a, const int32_t* pairs, const NearUnit* units, int nunits, int nrhs,
                             C2<T>* y, int64_t n, cudaStream_t st) {
  if (nunits <= 0) return;
  rhs_chunks<T, 8>(nrhs, [&](auto w, int rh, int nr) {
    mv_backward_leaf<T, decltype(w)::value>
        <<<chunk_grid<decltype(w)::value>(nunits, nr), 128, 0, st>>>(a, pairs, units, rh, nr, nrhs, y, n);
  });
}
template <typename T>
void launch_mv_near(const MvArgs<T>& a, bool adj, int nrhs, const C2<T>* x, C2<T>* y, int64_t n,
                    const int32_t* pairs, const NearUnit* leafs, int nleafs, cudaStream_t st) {
  const int grid = a.nunits + nleafs;
  if (grid <= 0) return;
  // FP64, bound by its pipe: as narrow chunks as give every SM two CTAs (reading
  // the matrix, then small, again from L2).  n = 400, seven vectors: 54 -> 25 us;
  // two: 22 -> 18
  int most = 8;
  while (sizeof(T) == 8 && most > 1 && (int64_t)grid * ((nrhs + most - 1) / most) < 2 * 152) most /= 2;
  if (most < 8 && nrhs % most != 0) most = 1;  // one launch instead of two, each of too few CTAs
  rhs_chunks<T, 8>(nrhs, [&](auto w, int rh, int nr) {
    constexpr int NR = decltype(w)::value;
    if (adj) mv_near<T, NR, true><<<chunk_grid<NR>(grid, nr), 128, 0, st>>>(a, rh, nr, x, y, n, pairs, leafs, nrhs);
    else mv_near<T, NR, false><<<chunk_grid<NR>(grid, nr), 128, 0, st>>>(a, rh, nr, x, y, n, pairs, leafs, nrhs);
  }, most);
}

#define DH2_MV_INST(T)                                                                                      \
  template void launch_mv_forward_leaf<T>(const SideView<T>&, const int32_t*, int, const C2<T>*, int,      \
                                          int64_t, C2<T>*, const int64_t*, C2<T>*, cudaStream_t);          \
  template void launch_mv_forward_up<T>(const SideView<T>&, const int32_t*, int, int, C2<T>*,              \
                                        const int64_t*, cudaStream_t);                                     \
  template void launch_mv_coupling<T>(const MvArgs<T>&, int, int, cudaStream_t);                           \
  template void launch_mv_coupling_adj<T>(const MvArgs<T>&, int, int, cudaStream_t);                       \
  template void launch_mv_backward_down<T>(const MvArgs<T>&, const int32_t*, int, int, cudaStream_t);      \
  template void launch_mv_backward_leaf<T>(const MvArgs<T>&, const int32_t*, const NearUnit*, int, int,    \
                                           C2<T>*, int64_t, cudaStream_t);                                 \
  template void launch_mv_near<T>(const MvArgs<T>&, bool, int, const C2<T>*, C2<T>*, int64_t, const int32_t*, \
                                  const NearUnit*, int, cudaStream_t);
DH2_MV_INST(float)
DH2_MV_INST(double)

}  // namespace dh2

// Device-side types and kernel entry points of the compression library.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace dh2 {

template <typename T>
struct __align__(2 * sizeof(T)) C2 {
  T re, im;
};

// Arguments of the per-pair factorisation kernel (one CTA per (cluster,
// direction) pair).  Index [side] selects the row (0) or column (1) basis.
// Launch choices the autotuner sets (the public dh2_tuning, validated): one
// table per process, read when a compression prepares its launches.
struct TuneTable {
  int32_t jacobi_tpp[5];     // factor classes (<= 32, 40, 48, 64 rows, more): most threads per Jacobi column pair
  int32_t jacobi_narrow[4];  // FP32 and mixed leaf classes: Jacobi CTAs of ~4 (0), ~2 (1) or ~1 (2) x rows threads
  int32_t rq_ctas_per_sm;    // leaf R kernel: resident CTAs per SM (0: its occupancy limit)
  int32_t rq_tensor;         // mixed mode: leaf R on the tensor cores (1) or the FP32 pipes (0)
  int32_t level_seg_cols;    // non-leaf pairs wider than twice this: factored by column segments (0: never)
};
TuneTable tune_current();
// factor class of a pair kernel compiled for P_T rows
__host__ __device__ constexpr int factor_class(int P_T) {
  return P_T <= 32 ? 0 : P_T <= 40 ? 1 : P_T <= 48 ? 2 : P_T <= 64 ? 3 : 4;
}

// ---------------------------------------------------------------- generated entries
// Entry G_ij generated from the points, with `diag` on the diagonal:
//  - without normals: the Helmholtz single layer of Eq. (helmholtz),
//    exp(i kappa r) / (4 pi r), r = |x_i - x_j|;
//  - otherwise the double layer of Section 7 ("DLP matrix"),
//    (1 - i kappa r) exp(i kappa r) / (4 pi r^3) <x_i - x_j, n(x_j)>.
template <typename T>
struct Gen;

// FP64: points and unit normals (NULL: single layer), 3 doubles each.
template <>
struct Gen<double> {
  const double* pts;
  const double* nrm;
  double kappa, diag;
};
__device__ __forceinline__ C2<double> gen_entry(const Gen<double>& g, int64_t i, int64_t j) {
  if (i == j) return C2<double>{g.diag, 0.0};
  const double dx = g.pts[3 * i] - g.pts[3 * j];
  const double dy = g.pts[3 * i + 1] - g.pts[3 * j + 1];
  const double dz = g.pts[3 * i + 2] - g.pts[3 * j + 2];
  const double r = sqrt(dx * dx + dy * dy + dz * dz);
  // single layer: scale 1/(4 pi r); double layer: <x_i - x_j, n_j>/(4 pi r^3)
  // times (1 - i kappa r)
  double scale;
  double kr = 0.0;
  if (g.nrm) {
    const double dn = dx * g.nrm[3 * j] + dy * g.nrm[3 * j + 1] + dz * g.nrm[3 * j + 2];
    scale = dn / (12.566370614359172 * r * r * r);
    kr = g.kappa * r;
  } else {
    scale = 1.0 / (12.566370614359172 * r);
  }
  double sn, cs;
  sincos(g.kappa * r, &sn, &cs);
  // (cs + i sn)(1 - i kr) = cs + kr sn + i (sn - kr cs)
  return C2<double>{(cs + kr * sn) * scale, (sn - kr * cs) * scale};
}

// A value hi + lo of two floats (|lo| <= ulp(hi)/2, about 48 significant
// bits), with the error-free sum of Knuth and the error-free product from a
// fused multiply-add (Dekker's double-length arithmetic in FP32 registers).
struct Df {
  float hi, lo;
};
__device__ __forceinline__ Df df_fast_sum(float s, float e) {  // |s| >= |e|
  const float h = __fadd_rn(s, e);
  return Df{h, __fsub_rn(e, __fsub_rn(h, s))};
}
__device__ __forceinline__ Df df_add(Df x, Df y) {
  const float s = __fadd_rn(x.hi, y.hi);
  const float bb = __fsub_rn(s, x.hi);
  const float e = (__fsub_rn(x.hi, __fsub_rn(s, bb)) + __fsub_rn(y.hi, bb)) + x.lo + y.lo;
  return df_fast_sum(s, e);
}
__device__ __forceinline__ Df df_neg(Df x) { return Df{-x.hi, -x.lo}; }
__device__ __forceinline__ Df df_mul(Df x, Df y) {
  const float p = __fmul_rn(x.hi, y.hi);
  float e = fmaf(x.hi, y.hi, -p);
  e = fmaf(x.hi, y.lo, e);
  e = fmaf(x.lo, y.hi, e);
  return df_fast_sum(p, e);
}
// unnormalised forms: a leading float and the sum of the errors behind it
struct Df2 {
  float p, e;
};
__device__ __forceinline__ Df2 two_sum(float x, float y) {
  const float s = __fadd_rn(x, y), bb = __fsub_rn(s, x);
  return Df2{s, __fadd_rn(__fsub_rn(x, __fsub_rn(s, bb)), __fsub_rn(y, bb))};
}
__device__ __forceinline__ Df2 df_sq(Df x) {
  const float p = __fmul_rn(x.hi, x.hi);
  return Df2{p, fmaf(2.f * x.hi, x.lo, fmaf(x.hi, x.hi, -p))};
}
__device__ __forceinline__ Df2 df_prod(Df x, Df y) {
  const float p = __fmul_rn(x.hi, y.hi);
  return Df2{p, fmaf(x.lo, y.hi, fmaf(x.hi, y.lo, fmaf(x.hi, y.hi, -p)))};
}
__device__ __forceinline__ Df df_diff(float xh, float xl, float yh, float yl) {
  const Df2 s = two_sum(xh, -yh);
  return df_fast_sum(s.p, s.e + __fsub_rn(xl, yl));
}
__device__ __forceinline__ Df df_split(double v) {
  const float h = (float)v;
  return Df{h, (float)(v - (double)h)};
}

// FP32: coordinates, relative to the middle of their bounding box and to a power
// of two above its extent, (and normals) split into two floats each, per point
// two (with normals four) float4: hi parts, lo parts.  Differences, r, the phase
// and its reduction are formed in double-float, sin and cos of the reduced
// phase in FP32, while that leaves an entry's error to its FP32 roundings.  It
// does not where a difference cancels: a coordinate difference is off by up to
// 2^-49 (of the scaled extent), <x_i - x_j, n_j> by 2^-48 + 2^-45.5 r.  Entries
// with r or |<x_i - x_j, n_j>| below 2^22 times that, and all of them where the
// scaled quantities leave the range (near2 infinite), are formed from the FP64
// points as in the FP64 form (gen_entry_f64): rare on a surface mesh (spacing
// above 2^-21 of its extent), but one in six entries on a flat face of a double
// layer, most of those exactly zero.  GB300's narrow FP64 pipe (about 2 lanes per SM
// against 128) had made FP64 differences and phases for every entry most of the
// matrix-free mode's time.  n = 16384 cube, before -> after: norms and nearfield
// 14.9 -> 1.7 ms, leaf R 4.7 -> 0.9 ms, leaf factors 11.5 -> 7.8 ms (the whole
// compression 32.3 -> 7.7 ms, 8.0 with the tests for cancellation; double layer
// 42.9 -> 10.7 ms).
template <>
struct Gen<float> {
  const float4* pts;
  int dlp;       // with normals
  Df ppi, kap;   // kappa / pi, kappa, for the scaled points
  float diag;
  float scale;   // of the entries: the points' factor (double layer: its square)
  float near2;   // entries with r^2 below this go by the FP64 points
  Gen<double> g64;
};
// An entry from the FP64 points: differences, distance, phase and its reduction
// in FP64, sin and cos of the reduced phase in FP32.  (Arguments by value: by
// reference the callers' copies went through local memory.)
static __device__ __noinline__ C2<float> gen_entry_f64(const Gen<double> g, int i, int j) {
  const double *x = g.pts + 3 * (int64_t)i, *y = g.pts + 3 * (int64_t)j;
  const double dx = x[0] - y[0], dy = x[1] - y[1], dz = x[2] - y[2];
  double dn = 0.0;
  if (g.nrm) {
    const double* v = g.nrm + 3 * (int64_t)j;
    const double nx = v[0], ny = v[1], nz = v[2];
    // an axis-parallel flat face: every product is an exact zero (two points at one place: below)
    if ((dx == 0.0 || nx == 0.0) && (dy == 0.0 || ny == 0.0) && (dz == 0.0 || nz == 0.0) &&
        (dx != 0.0 || dy != 0.0 || dz != 0.0))
      return C2<float>{0.f, 0.f};
    dn = dx * nx + dy * ny + dz * nz;
  }
  const double r = sqrt(dx * dx + dy * dy + dz * dz), kr = g.kappa * r;
  const float sc = (float)(g.nrm ? dn / (12.566370614359172 * r * r * r) : 1.0 / (12.566370614359172 * r));
  double th = kr * 0.31830988618379067;  // phase / pi
  th -= 2.0 * rint(0.5 * th);            // reduced to [-1, 1]
  float sn, cs;
  sincospif((float)th, &sn, &cs);
  const float k = g.nrm ? (float)kr : 0.f;
  return C2<float>{fmaf(k, sn, cs) * sc, fmaf(-k, cs, sn) * sc};
}
__device__ __forceinline__ C2<float> gen_entry(const Gen<float>& g, int64_t i, int64_t j) {
  if (i == j) return C2<float>{g.diag, 0.f};
  const int st = g.dlp ? 4 : 2;
  const float4 *pi = g.pts + i * st, *pj = g.pts + j * st;
  const float4 xh = __ldg(pi), xl = __ldg(pi + 1), yh = __ldg(pj), yl = __ldg(pj + 1);
  const Df dx = df_diff(xh.x, xl.x, yh.x, yl.x);
  const Df dy = df_diff(xh.y, xl.y, yh.y, yl.y);
  const Df dz = df_diff(xh.z, xl.z, yh.z, yl.z);
  // |x_i - x_j|^2: the products' and the sums' errors gathered in one float
  const Df2 sx = df_sq(dx), sy = df_sq(dy), sz = df_sq(dz);
  const Df2 s1 = two_sum(sx.p, sy.p), s2 = two_sum(s1.p, sz.p);
  const Df d2 = df_fast_sum(s2.p, ((sx.e + sy.e) + sz.e) + (s1.e + s2.e));
  if (!(d2.hi >= g.near2)) return gen_entry_f64(g.g64, (int)i, (int)j);
  // r = sqrt(d2): one Newton step from the FP32 square root
  const float ir = rsqrtf(d2.hi), r0 = __fmul_rn(d2.hi, ir);
  const float rest = fmaf(-r0, r0, d2.hi) + d2.lo;
  const Df r = df_fast_sum(r0, 0.5f * ir * rest);
  // phase / pi, reduced to [-1, 1]: the integer part leaves the leading float exactly
  const Df2 ph = df_prod(r, g.ppi);
  const float th = __fsub_rn(ph.p, 2.f * rintf(0.5f * ph.p)) + ph.e;
  float sn, cs;
  sincospif(th, &sn, &cs);
  const Df2 q4 = df_prod(r, Df{12.566371f, -8.742278e-7f});  // 4 pi r
  if (!g.dlp) {  // 1 / (4 pi r), the quotient corrected by its remainder
    const float s0 = ir * 0.07957747f;
    const float sc = fmaf(s0, fmaf(-s0, q4.p, 1.f) - s0 * q4.e, s0) * g.scale;
    return C2<float>{cs * sc, sn * sc};
  }
  const float4 nh = __ldg(pj + 2), nl = __ldg(pj + 3);
  const Df dn = df_add(df_add(df_mul(dx, Df{nh.x, nl.x}), df_mul(dy, Df{nh.y, nl.y})), df_mul(dz, Df{nh.z, nl.z}));
  if (fabsf(dn.hi) < fmaf(0x1p-19f, r.hi, 0x1p-21f)) return gen_entry_f64(g.g64, (int)i, (int)j);
  const Df q = df_mul(df_fast_sum(q4.p, q4.e), d2);
  const float iq = __frcp_rn(q.hi), s0 = dn.hi * iq;
  const float sc = fmaf((fmaf(-s0, q.hi, dn.hi) + dn.lo) - s0 * q.lo, iq, s0) * g.scale;
  const Df kr = df_mul(r, g.kap);
  return C2<float>{fmaf(kr.hi, sn, cs) * sc, fmaf(-kr.hi, cs, sn) * sc};
}

template <typename T>
struct PairArgs {
  const int32_t* start[2];            // first row index of the pair's cluster
  const int32_t* m[2];                // leaf rows (cluster size)
  const int32_t* ncols[2];            // #F_tc
  const int64_t* cmoff[2];            // leaf column-map offsets
  const int32_t* gcol[2];             // leaf column map: index of G's other dimension
  const int32_t* gblk[2];             // leaf column map: block id
  const T* colw[2];                   // leaf column map: weight 1/omega of the column's block
  const int32_t* son[2];              // non-leaf: 2 son pairs
  const int32_t* sonoff[2];           // non-leaf: column offsets in the son pairs
  const int32_t* level[2];
  const int32_t* kcap[2];             // rank capacity = leading dimension of R
  const int32_t* rowcap[2];           // leading dimension of the stored Q / [E1;E2]
  const int64_t* Roff[2];
  const int64_t* Qoff[2];
  const C2<T>* G;
  int64_t ld;
  const double* invw;                 // per block 1/omega_b
  C2<T>* R[2];
  C2<T>* Q[2];
  double* sig[2];                     // per pair P values (descending)
  int32_t* rank[2];
  const double* eps2;                 // per level eps_l^2
  float4* H;                          // FP32 and mixed modes: leaf Gram matrices (see GramArgs)
  float4* L4;                         // and leaf Cholesky factors, pair at L4 + its Gram offset (FP32 complex, ld p)
  // per pair, first entry of its Gram matrix: a leaf pair's in H, a non-leaf
  // pair's (one per column segment, mp x mp each) in Hl, from its level's start
  const int64_t* hoff[2];
  float4* Hl;
  const int32_t* gseg_cols;           // per level: columns of a non-leaf pair's Gram segment
  const int32_t* rank_ovr[2];         // per pair a rank replacing the truncation rule (< 0: the rule), or NULL
  int32_t max_sweeps;
  int32_t jacobi_tpp[5];              // per factor class: most threads per Jacobi column pair (TuneTable)
  // non-leaf pairs factored by column segments: per pair the first entry of
  // its segments' factors in seg_buf (p x p each, ld p, one after the other),
  // -1 if not split; seg_cols columns per segment
  const int64_t* seg_off[2];
  C2<T>* seg_buf;
  int32_t seg_cols;
  uint32_t* status;
  Gen<T> entry;  // matrix-free mode (gen != 0): entries generated from points
  int32_t gen;
};

// One CTA per launch code: args_dev holds one PairArgs per problem (device
// memory); P is the row capacity of the shared-memory factor (even).  With
// `count` (device int) the launch is sized at capacity nblocks and CTAs at or
// past *count return at once, so a list whose length is known only on the
// device needs no read-back.  Returns false, launching nothing, if the shared
// memory the launch needs exceeds the device's per-block limit.  With `segs`
// (non-leaf pairs only; codes unused) each CTA takes an entry code << 32 |
// segment and forms that column segment's LQ factor into the pair's slot of
// the segment buffer.
template <typename T>
bool launch_pair_kernel(const PairArgs<T>* args_dev, const uint32_t* codes, int nblocks, int P, bool from_r,
                        cudaStream_t st, const int* count = nullptr, const uint64_t* segs = nullptr);

// The factorisation from Gram matrices (FP32 and mixed modes, pairs of at most
// kGramRows rows): the pair kernel with steps 1 and 1b replaced by the pivoted
// Cholesky of H (launch_gram or launch_gram_i64 before it), then Jacobi, rank
// and Q.  Non-leaf pairs (from_r): H summed over the pair's column segments;
// count as for launch_pair_kernel.
constexpr int kGramRows = 64;
bool launch_gram_cholesky(const PairArgs<float>* args_dev, const uint32_t* codes, int nblocks, int P, bool from_r,
                          cudaStream_t st, const int* count = nullptr);
bool launch_gram_jacobi(const PairArgs<float>* args_dev, const uint32_t* codes, int nblocks, int P, bool from_r,
                        cudaStream_t st, const int* count = nullptr);

// H = A A^* from products of fixed-point integers on the integer pipe, FP32
// mode's leaf pairs (codes) or a level's pairs by segments of their level's
// gseg_cols columns (segs: code << 32 | segment; pairs above kGramRows rows are
// left to the LQ launches).  P: most rows of the list.  A level's segments are
// kGramSegCols columns wide, or the first doubling of that with at most
// kGramSegMax segments beside one per pair: a matrix of up to 64 KB each, so
// that the scratch stays a few hundred MB (n = 32768, paper's parameters, 256
// columns throughout: 3.3 GB) with some ten waves of CTAs.
constexpr int kGramSegCols = 256, kGramSegMax = 4096;
// seg_cols: of the segments, at most.
bool launch_gram_i64(const PairArgs<float>* args_dev, const uint32_t* codes, const uint64_t* segs, int n, int P,
                     int seg_cols, bool gen, cudaStream_t st);

// R = Q^* A for the pairs of a pair-kernel launch, after it, by tiles of 32
// columns, tiles[i] = launch code << 32 | first column (P as for the pair
// kernel).  Leaf tiles of a stored G (gen false) go to a persistent kernel
// that keeps the next tile's loads in flight; the others get one CTA per tile.
template <typename T>
bool launch_rq_kernel(const PairArgs<T>* args_dev, const uint64_t* tiles, int ntiles, int P, bool from_r, bool gen,
                      cudaStream_t st);

// Non-leaf codes of one level split by the row count of their Ghat (from the
// sons' ranks): out = 4 segments of n codes, counts[4] zeroed by the caller;
// merge: the pairs of at most kGramRows rows all in segment 2.
template <typename T>
void launch_classify(const PairArgs<T>* args_dev, const uint32_t* codes, int n, uint32_t* out, int* counts, bool merge,
                     cudaStream_t st);
// the same for segment entries (code << 32 | segment)
template <typename T>
void launch_classify_seg(const PairArgs<T>* args_dev, const uint64_t* segs, int n, uint64_t* out, int* counts,
                         cudaStream_t st);

// *out = the problems' status words combined (n <= kMaxBatch)
template <typename T>
void launch_status_or(const PairArgs<T>* args_dev, int n, uint32_t* out, cudaStream_t st);

// Arguments of the leaf Gram kernel of the mixed modes (one per problem).
// Index [side] selects the row (0) or column (1) basis.
struct GramArgs {
  const int32_t* start[2];   // first row index of the pair's cluster
  const int32_t* m[2];       // leaf rows
  const int32_t* ncols[2];   // #F_tc
  const int64_t* cmoff[2];   // leaf column-map offsets
  const int32_t* gcol[2];    // leaf column map: index of G's other dimension
  const float* colw[2];      // leaf column map: weight 1/omega of the column's block
  const int64_t* hoff[2];    // per pair: first entry of its Gram in H (mp x mp, mp = m rounded up to 8)
  const int64_t* seg_begin[2];  // per pair: its blocks of F_tc as a range of column-map segments
  const int32_t* seg_blk[2];    // per segment: block id
  const int32_t* bt;         // per block: row cluster
  const int32_t* bs;         // per block: column cluster
  const int32_t* cstart;     // per cluster: first index
  const int32_t* csize;      // per cluster: size
  const double* invw;        // per block: 1/omega_b
  const float* bmax;         // per admissible block: largest |re|, |im| per row, then per column
  const int64_t* bmax_off;
  const C2<float>* G;
  int64_t ld;
  float4* H;                 // Gram matrices: (re hi, re lo, im hi, im lo) double-float, column-major, ld mp
  uint32_t* status;
  uint32_t spin_limit;       // polls of a wait for a tensor-core batch (0: default)
};
// Columns of one exact accumulation window of the Gram kernel.
constexpr int kGramWindow = 448;

// H = A A^* for the leaf pairs of a launch list (leaves of at most maxm <= 64
// rows) on the tensor cores; false if the launch cannot run.
bool launch_gram(const GramArgs* args_dev, const uint32_t* codes, int n, int maxm, cudaStream_t st);

// R = Q^* A of the mixed mode's leaf pairs on the tensor cores, over a list of
// R tiles of kRTile columns (all leaf classes; a 128-column tile starts at
// every entry whose first column is a multiple of 128); false if it cannot run.
bool launch_rq_tc(const PairArgs<float>* args_dev, const uint64_t* tiles, int64_t ntiles, uint32_t spin_limit,
                  cudaStream_t st);

// Phase cycle counters of the pair kernel (only with -DDH2_PROFILE); 17 values.
void prof_reset_pair();
bool prof_read_pair(unsigned long long* out17);
// Phase cycle counters of the Gram kernels (only with -DDH2_PROFILE): 10
// values of the one-stage form, then 12 of the pipelined form.
void prof_reset_gram();
bool prof_read_gram(unsigned long long* out22);

}  // namespace dh2

// Galerkin product A_c = P^T A P on rectangular-block matrices (Sec. 2.2,
// Sec. 3.1): symbolic phase once (host), numeric phase reused (device).
//
// Numeric design.  Stage 1 computes the intermediate Z = A P, one output block
// per lane group (bs_p lanes, one per output column): each lane accumulates
// its column over the block pairs (A_ik, P_kJ) in the output's gather list.
// Stage 2 computes A_c = P^T Z the same way over the pairs (P_iI, Z_iJ).
// Lists are fixed by the symbolic phase, so results are deterministic and no
// atomics are used.  The gather lists keep every FMA useful (no padding to dense
// local blocks).  The FP64 pipe, at 2 FMA/clock/SM, would take 4.0 ms for the
// finest level's product at 64^3; four of nine products run there and the rest
// in fixed point on the integer pipes (fixed.cuh), from operands cut once per
// block instead of once per pair (64^3: stage 1 2.86 -> 1.85 ms with the cut,
// stage 2 1.21 -> 0.70).  Stage 1 takes its items in runs of a
// row, so that a warp's lane groups share the row's A blocks; stage 2 in
// windows ordered by work, a long list shared by up to eight warps.
#include <algorithm>
#include <numeric>

#include "device.cuh"
#include "internal.h"

namespace bamg {

// Values of a block in the FP32 stages' block-ordered copies: padded to whole
// 16-byte words, so that a block's values come in a quarter of the loads (the
// stages are bound by L1's rate of scattered loads: 51^3, stage 1 462 -> 420 us
// with the copy, stage 2 215 -> 183).  The FP64 copies of P stay unpadded.
template <typename T>
__host__ __device__ constexpr int block_pitch(int n) { return sizeof(T) == 4 ? (n + 3) / 4 * 4 : n; }

template <int N>
__device__ __forceinline__ void load_block(const float* __restrict__ p, float (&v)[N]) {
#pragma unroll
  for (int k = 0; k < (N + 3) / 4; ++k) {
    const float4 q = __ldg(reinterpret_cast<const float4*>(p) + k);
    const float w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (4 * k + e < N) v[4 * k + e] = w[e];
  }
}

// Column c of the sum over the list entries [s0, s1) of A_ik P_kJ (FP32).
template <int BS, int BSP>
__device__ __forceinline__ void stage1_column32(int s0, int s1, const int* __restrict__ ea,
                                                const int* __restrict__ ep, const float* __restrict__ Ablk,
                                                const float* __restrict__ Pblk, int c, float (&acc)[BS]) {
#pragma unroll
  for (int r = 0; r < BS; ++r) acc[r] = 0.0f;
#pragma unroll 2
  for (int s = s0; s < s1; ++s) {
    const int64_t aslot = __ldg(ea + s);
    const int64_t pb = __ldg(ep + s);
    float a[BS * BS], p[BS];
    load_block<BS * BS>(Ablk + aslot * block_pitch<float>(BS * BS), a);
#pragma unroll
    for (int q = 0; q < BS; ++q) p[q] = __ldg(Pblk + pb * block_pitch<float>(BS * BSP) + q * BSP + c);
#pragma unroll
    for (int r = 0; r < BS; ++r)
#pragma unroll
      for (int q = 0; q < BS; ++q) acc[r] = fma(a[r * BS + q], p[q], acc[r]);
  }
}

// Column c of the sum of P_iI^T Z_iJ (FP32).
template <int BS, int BSP>
__device__ __forceinline__ void stage2_column32(int s0, int s1, const int* __restrict__ ep,
                                                const int* __restrict__ ez, const float* __restrict__ Pblk,
                                                const float* __restrict__ Z, int c, float (&acc)[BSP]) {
#pragma unroll
  for (int u = 0; u < BSP; ++u) acc[u] = 0.0f;
#pragma unroll 2
  for (int s = s0; s < s1; ++s) {
    const int64_t pb = __ldg(ep + s);
    const int64_t z = __ldg(ez + s);
    float p[BS * BSP], zc[BS];
    load_block<BS * BSP>(Pblk + pb * block_pitch<float>(BS * BSP), p);
#pragma unroll
    for (int r = 0; r < BS; ++r) zc[r] = __ldg(Z + z * (BS * BSP) + r * BSP + c);
#pragma unroll
    for (int r = 0; r < BS; ++r)
#pragma unroll
      for (int u = 0; u < BSP; ++u) acc[u] = fma(p[r * BSP + u], zc[r], acc[u]);
  }
}

// The same columns by FP64 FMA, from the sliced storage.
template <int BS, int BSP, typename T>
__device__ __forceinline__ void stage1_column(int s0, int s1, const int* __restrict__ ea, const int* __restrict__ ep,
                                              const T* __restrict__ Avals, const T* __restrict__ Pblk, int c,
                                              T (&acc)[BS]) {
#pragma unroll
  for (int r = 0; r < BS; ++r) acc[r] = T(0);
  for (int s = s0; s < s1; ++s) {
    const int64_t aslot = __ldg(ea + s);
    const int64_t pb = __ldg(ep + s);
    T p[BS];
#pragma unroll
    for (int q = 0; q < BS; ++q) p[q] = __ldg(Pblk + pb * (BS * BSP) + q * BSP + c);
    const T* a = Avals + (aslot >> 5) * (32LL * BS * BS) + (aslot & 31);
#pragma unroll
    for (int r = 0; r < BS; ++r)
#pragma unroll
      for (int q = 0; q < BS; ++q) acc[r] = fma(__ldg(a + 32 * (r * BS + q)), p[q], acc[r]);
  }
}

template <int BS, int BSP, typename T>
__device__ __forceinline__ void stage2_column(int s0, int s1, const int* __restrict__ ep, const int* __restrict__ ez,
                                              const T* __restrict__ Pblk, const T* __restrict__ Z, int c,
                                              T (&acc)[BSP]) {
#pragma unroll
  for (int u = 0; u < BSP; ++u) acc[u] = T(0);
  for (int s = s0; s < s1; ++s) {
    const int64_t pb = __ldg(ep + s);
    const int64_t z = __ldg(ez + s);
    T zc[BS];
#pragma unroll
    for (int r = 0; r < BS; ++r) zc[r] = __ldg(Z + z * (BS * BSP) + r * BSP + c);
    const T* p = Pblk + pb * (BS * BSP);
#pragma unroll
    for (int r = 0; r < BS; ++r)
#pragma unroll
      for (int u = 0; u < BSP; ++u) acc[u] = fma(__ldg(p + r * BSP + u), zc[r], acc[u]);
  }
}

// Products of a block that the FP64 stages leave on the FP64 pipe (fixed.cuh):
// four of nine from 3-row blocks (64^3, four, five, six of nine: stage 1 with the
// cut 1.85, 2.01, 2.29 ms, stage 2 0.70, 0.72, 0.85), three of nine for 6x6
// blocks (MIS hierarchy at 48^3, both its products, two, three, four, five, six:
// stage 1 4.95, 4.01, 4.24, 4.61, 5.20 ms; stage 2 1.25, 1.34, 1.53, 1.75 with
// three to six).
constexpr int stage1_fma(int bs) { return bs * bs * (bs == 3 ? 4 : 3) / 9; }
constexpr int stage2_fma(int bs, int bsp) { return bs * bsp * (bs == 3 ? 4 : 3) / 9; }
// CTAs of 256 threads per SM that the FP64 stages are held to.  3-row blocks: 64
// and 80 registers, where the compiler would take 74 and 96 and leave 24 and 16
// warps per SM to cover the lists' chains of loads; 6x6: 128, where it would take
// 152 and leave one CTA (stage 2 of the 48^3 example 1.97 ms so).
template <int BS, typename T>
constexpr int kStage1Ctas = sizeof(T) == 8 ? (BS == 3 ? 4 : 2) : 0;
template <int BS, typename T>
constexpr int kStage2Ctas = sizeof(T) == 8 ? (BS == 3 ? 3 : 2) : 0;
template <int BS>
using ACut = FxCut<BS, BS, stage1_fma(BS)>;
template <int BS, int BSP>
using PCut = FxCut<BSP, BS, stage2_fma(BS, BSP)>;  // of the transposed block

// The same columns with FP64 products on both pipes (fixed.cuh); false where
// the values are not covered and the forms above have to be taken.  The six
// lanes of an output block share A_ik (stage 1) and P_iI (stage 2), so these
// are read cut, from block-ordered copies: a lane that cut A_ik itself read it
// as nine sectors of the sliced storage and repeated the others' work.  The
// next pair's numbers are requested before this one's products.
template <int BS, int BSP>
__device__ __forceinline__ bool stage1_column_fx(int s0, int s1, const int* __restrict__ ea,
                                                 const int* __restrict__ ep, const uint4* __restrict__ Acut,
                                                 const double* __restrict__ Pblk, int c, double (&acc)[BS]) {
  using Cut = ACut<BS>;
  constexpr int F0 = stage1_fma(BS);
  FxSum<BS, BS, F0> sum;
  sum.init();
  int ia = s0 < s1 ? __ldg(ea + s0) : 0, ib = s0 < s1 ? __ldg(ep + s0) : 0;
#pragma unroll 1
  for (int s = s0; s < s1; ++s) {
    const uint4* pa = Acut + (int64_t)ia * Cut::kWords;
    const double* pp = Pblk + (int64_t)ib * (BS * BSP) + c;
    if (s + 1 < s1) {
      ia = __ldg(ea + s + 1);
      ib = __ldg(ep + s + 1);
    }
    double f[F0], p[BS];
    typename Cut::Block a;
    Cut::load(pa, f, a);
#pragma unroll
    for (int q = 0; q < BS; ++q) p[q] = __ldg(pp + q * BSP);
    sum.add([&](int r, int q) { return f[r * BS + q]; }, a, p);
  }
  return sum.finish(acc);
}

template <int BS, int BSP>
__device__ __forceinline__ bool stage2_column_fx(int s0, int s1, const int* __restrict__ ep,
                                                 const int* __restrict__ ez, const uint4* __restrict__ Pcut,
                                                 const double* __restrict__ Z, int c, double (&acc)[BSP]) {
  using Cut = PCut<BS, BSP>;
  constexpr int F0 = stage2_fma(BS, BSP);
  FxSum<BSP, BS, F0> sum;
  sum.init();
  int ib = s0 < s1 ? __ldg(ep + s0) : 0, iz = s0 < s1 ? __ldg(ez + s0) : 0;
#pragma unroll 1
  for (int s = s0; s < s1; ++s) {
    const uint4* pp = Pcut + (int64_t)ib * Cut::kWords;
    const double* pz = Z + (int64_t)iz * (BS * BSP) + c;
    if (s + 1 < s1) {
      ib = __ldg(ep + s + 1);
      iz = __ldg(ez + s + 1);
    }
    double f[F0], zc[BS];
    typename Cut::Block p;
    Cut::load(pp, f, p);
#pragma unroll
    for (int r = 0; r < BS; ++r) zc[r] = __ldg(pz + r * BSP);
    sum.add([&](int u, int r) { return f[u * BS + r]; }, p, zc);
  }
  return sum.finish(acc);
}

// Cut copies: A's blocks by storage slot, and P's blocks transposed, in block
// order.  A lane packs a block; the warp writes its 32 blocks as one run.
template <int W>
__device__ __forceinline__ void write_cut(const uint4 (&w)[W], int64_t first, int64_t n, uint4* stage,
                                          uint4* __restrict__ out) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < W; ++k) stage[lane * W + k] = w[k];
  __syncwarp();
  for (int k = lane; k < (int)min((int64_t)32, n - first) * W; k += 32) out[first * W + k] = stage[k];
}

template <int BS>
__global__ void __launch_bounds__(64) k_cut_slots(int64_t nslots, const double* __restrict__ vals,
                                                  uint4* __restrict__ out) {
  using Cut = ACut<BS>;
  __shared__ uint4 stage[2][32 * Cut::kWords];
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nslots) return;  // whole warps
  double v[BS * BS];
#pragma unroll
  for (int e = 0; e < BS * BS; ++e) v[e] = __ldcs(vals + vidx<BS * BS>(t, e));
  uint4 w[Cut::kWords];
  Cut::pack([&](int r, int q) { return v[r * BS + q]; }, w);
  write_cut<Cut::kWords>(w, t & ~31LL, nslots, stage[threadIdx.x >> 5], out);
}

// FP32 blocks by storage slot, padded (block_pitch).
template <int BS>
__global__ void __launch_bounds__(128) k_pad_slots(int64_t nslots, const float* __restrict__ vals,
                                                   float4* __restrict__ out) {
  constexpr int N = BS * BS, W = block_pitch<float>(N) / 4;
  __shared__ float4 stage[4][32 * W];
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nslots) return;  // whole warps
  float v[4 * W];
#pragma unroll
  for (int e = 0; e < 4 * W; ++e) v[e] = e < N ? __ldcs(vals + vidx<N>(t, e)) : 0.0f;
  const int lane = threadIdx.x & 31;
  float4* mine = stage[threadIdx.x >> 5];
#pragma unroll
  for (int k = 0; k < W; ++k) mine[lane * W + k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
  __syncwarp();
#pragma unroll
  for (int k = 0; k < W; ++k) out[(t - lane) * W + k * 32 + lane] = mine[k * 32 + lane];
}

// FP32 blocks in block order, padded, from the FP64 ones.
__global__ void k_pad_blocks(int64_t nblk, int n, int pitch, const double* __restrict__ src, float* __restrict__ dst) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nblk * pitch) return;
  const int64_t b = t / pitch;
  const int e = (int)(t - b * pitch);
  dst[t] = e < n ? (float)src[b * n + e] : 0.0f;
}

template <int BS, int BSP>
__global__ void __launch_bounds__(64) k_cut_transposed(int64_t nblk, const double* __restrict__ Pblk,
                                                       uint4* __restrict__ out) {
  using Cut = PCut<BS, BSP>;
  __shared__ uint4 stage[2][32 * Cut::kWords];
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t first = t & ~31LL;
  if (first >= nblk) return;  // whole warps
  const int64_t b = min(t, nblk - 1);
  double v[BSP * BS];
#pragma unroll
  for (int r = 0; r < BS; ++r)
#pragma unroll
    for (int u = 0; u < BSP; ++u) v[u * BS + r] = __ldg(Pblk + b * (BS * BSP) + r * BSP + u);
  uint4 w[Cut::kWords];
  Cut::pack([&](int u, int r) { return v[u * BS + r]; }, w);
  write_cut<Cut::kWords>(w, first, nblk, stage[threadIdx.x >> 5], out);
}

template <int BS, int BSP, typename T>
__global__ void __launch_bounds__(256, kStage1Ctas<BS, T>) k_ptap_stage1(int64_t n1, int rounds, const int* __restrict__ item_z,
                                                     const int* __restrict__ off, const int* __restrict__ ea,
                                                     const int* __restrict__ ep, const T* __restrict__ Avals,
                                                     const T* __restrict__ Pblk, const uint4* __restrict__ Acut,
                                                     T* __restrict__ Z) {
  constexpr int G = 32 / BSP;
  const int lane = threadIdx.x & 31;
  const int g = lane / BSP, c = lane - g * BSP;
  if (g >= G) return;
  const int64_t first = (int64_t)blockIdx.x * rounds * 8 * G;
  for (int t = 0; t < rounds; ++t) {
    const int64_t item = first + (t * 8 + (threadIdx.x >> 5)) * G + g;
    if (item >= n1) return;
    T acc[BS];
    const int s0 = __ldg(off + item), s1 = __ldg(off + item + 1);
    if constexpr (std::is_same<T, double>::value) {
      if (!stage1_column_fx<BS, BSP>(s0, s1, ea, ep, Acut, Pblk, c, acc))
        stage1_column<BS, BSP, T>(s0, s1, ea, ep, Avals, Pblk, c, acc);
    } else {
      stage1_column32<BS, BSP>(s0, s1, ea, ep, Avals, Pblk, c, acc);
    }
    const int64_t z = __ldg(item_z + item);
#pragma unroll
    for (int r = 0; r < BS; ++r) Z[z * (BS * BSP) + r * BSP + c] = acc[r];
  }
}

// S warps share an item's list, each taking a run of it; their sums meet in
// shared memory and are added in list order (S = 1: no sharing).
template <int BS, int BSP, int S, typename T>
__global__ void __launch_bounds__(256, kStage2Ctas<BS, T>) k_ptap_stage2(int64_t n2, const int* __restrict__ item_slot,
                                                     const int* __restrict__ item_tslot,
                                                     const int* __restrict__ off, const int* __restrict__ ep,
                                                     const int* __restrict__ ez, const T* __restrict__ Pblk,
                                                     const uint4* __restrict__ Pcut, const T* __restrict__ Z,
                                                     T* __restrict__ Ac) {
  constexpr int G = 32 / BSP;
  constexpr int BC = BSP * BSP;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = warp % S;
  const int g = lane / BSP, c = lane - g * BSP;
  const int64_t item = ((int64_t)blockIdx.x * (8 / S) + warp / S) * G + g;
  const bool on = g < G && item < n2;
  T acc[BSP];
  if (on) {
    const int l0 = __ldg(off + item), l1 = __ldg(off + item + 1);
    const int part = (l1 - l0 + S - 1) / S;
    const int s0 = min(l1, l0 + sub * part), s1 = min(l1, s0 + part);
    if constexpr (std::is_same<T, double>::value) {
      if (!stage2_column_fx<BS, BSP>(s0, s1, ep, ez, Pcut, Z, c, acc))
        stage2_column<BS, BSP, T>(s0, s1, ep, ez, Pblk, Z, c, acc);
    } else {
      stage2_column32<BS, BSP>(s0, s1, ep, ez, Pblk, Z, c, acc);
    }
  }
  if constexpr (S > 1) {
    __shared__ T sums[8][BSP][32];
#pragma unroll
    for (int u = 0; u < BSP; ++u) sums[warp][u][lane] = on ? acc[u] : T(0);
    __syncthreads();
    if (!on) return;
    // each warp finishes components sub, sub + S, ...
#pragma unroll
    for (int u = 0; u < BSP; ++u) {
      if (u % S != sub) continue;
      T t = sums[warp - sub][u][lane];
#pragma unroll
      for (int k = 1; k < S; ++k) t += sums[warp - sub + k][u][lane];
      acc[u] = t;
    }
  }
  if (!on) return;
  const int64_t slot = __ldg(item_slot + item);
  T* o = Ac + (slot >> 5) * (32LL * BC) + (slot & 31);
  const int64_t ts = __ldg(item_tslot + item);
  T* tv = Ac + (ts >> 5) * (32LL * BC) + (ts & 31);
#pragma unroll
  for (int u = 0; u < BSP; ++u) {
    if (u % S != sub) continue;
    o[32 * (u * BSP + c)] = acc[u];
    if (ts >= 0) tv[32 * (c * BSP + u)] = acc[u];
  }
}

// Stage 1: items of one CTA, rounds x (8 warps x 32 / bs_p items).  A CTA takes a
// run of items in row order, sorted by list length, so that the items that
// share operand blocks (one row's and its neighbours') meet in one L1 while the
// lane groups of a warp still carry equal work; sorted over all items, every
// block comes from L2 or HBM once per list it is in (64^3: 2.27 -> 1.93 ms).
// More rounds share more but leave fewer CTAs: eight where each SM still gets
// eight CTAs.  Stage 2's lists differ too much in length within a
// run (0.63 ms sorted over all items, 1.07 in runs).
static int item_rounds(int64_t items, int bsp, int sm_count) {
  return (int)std::max<int64_t>(1, std::min<int64_t>(8, items / (8 * (32 / bsp) * sm_count * 8)));
}

// Stable order of items by decreasing list length within runs of `window`.
static std::vector<int> order_by_work(const std::vector<int>& off, int64_t window) {
  const int64_t n = (int64_t)off.size() - 1;
  std::vector<int> order((size_t)n);
  std::iota(order.begin(), order.end(), 0);
  for (int64_t w = 0; w < n; w += window)
    std::stable_sort(order.begin() + w, order.begin() + std::min(n, w + window),
                     [&](int a, int b) { return off[a + 1] - off[a] > off[b + 1] - off[b]; });
  return order;
}

// Reorder CSR-like lists (off, a, b) into item order.
static void permute_lists(const std::vector<int>& order, const std::vector<int>& off, const std::vector<int>& a,
                          const std::vector<int>& b, std::vector<int>& noff, std::vector<int>& na,
                          std::vector<int>& nb) {
  const size_t n = order.size();
  noff.assign(n + 1, 0);
  na.resize(a.size());
  nb.resize(b.size());
  for (size_t t = 0; t < n; ++t) {
    const int i = order[t];
    const int len = off[i + 1] - off[i];
    noff[t + 1] = noff[t] + len;
    std::copy(a.begin() + off[i], a.begin() + off[i + 1], na.begin() + noff[t]);
    std::copy(b.begin() + off[i], b.begin() + off[i + 1], nb.begin() + noff[t]);
  }
}

void ptap_release(bamg_ptap* p) {
  if (!p) return;
  cudaStream_t st = p->ctx->stream;
  dfree(p->s1_z, st);
  dfree(p->s1_off, st);
  dfree(p->s1_a, st);
  dfree(p->s1_p, st);
  dfree(p->s2_slot, st);
  dfree(p->s2_tslot, st);
  dfree(p->s2_off, st);
  dfree(p->s2_p, st);
  dfree(p->s2_z, st);
  dfree(p->Z, st);
  dfree(p->Z32, st);
  dfree(p->Pblk, st);
  dfree(p->Pblk32, st);
  ptap_trim(p);
  dfree(p->Apad, st);
}

void ptap_trim(bamg_ptap* p) {
  dfree(p->Acut, p->ctx->stream);
  dfree(p->Pcut, p->ctx->stream);
  p->pcut_version = ~0ull;
}

Status ptap_build(bamg_bsr* A, bamg_bsr* P, bool want_ac, bamg_ptap** plan_out, bamg_bsr** Ac_out) {
  *plan_out = nullptr;
  if (Ac_out) *Ac_out = nullptr;
  if (!A->has_pattern || !P->has_pattern) return make_status(BAMG_ERR_STATE, "Galerkin operands need patterns");
  if (A->br != A->bc || A->nbr != A->nbc)
    return make_status(BAMG_ERR_INVALID, "A must be square with square blocks");
  if (P->nbr != A->nbr || P->br != A->br)
    return make_status(BAMG_ERR_INVALID, "P rows (%lld x bs %d) do not match A (%lld x bs %d)", (long long)P->nbr,
                       P->br, (long long)A->nbr, A->br);
  const int bs = A->br, bsp = P->bc;
  const bool supported = (bs == 3 && bsp == 6) || (bs == 6 && bsp == 6) || (bs == 3 && bsp == 3);
  if (!supported) return make_status(BAMG_ERR_INVALID, "Galerkin block sizes %d -> %d not supported", bs, bsp);
  bamg_ctx* ctx = A->ctx;
  cudaStream_t st = ctx->stream;
  const int64_t n = A->nbr, nc = P->nbc;
  const auto &ar = A->h_rowptr, &ac = A->h_colidx, &aslot = A->h_slot_of;
  const auto &pr = P->h_rowptr, &pc = P->h_colidx;

  bamg_ptap* pl = new bamg_ptap();
  pl->ctx = ctx;
  pl->A = A;
  pl->P = P;
  pl->bs = bs;
  pl->bsp = bsp;
  pl->a_pid = A->pattern_id;
  pl->p_pid = P->pattern_id;
  pl->symmetric = A->symmetric;
  Status s = [&]() -> Status {
    // ---- Z = A P pattern and stage-1 lists (pairs in A-row order, then P-row order)
    std::vector<int>& zr = pl->h_zrowptr;
    std::vector<int>& zc = pl->h_zcol;
    zr.assign(n + 1, 0);
    std::vector<int> mark(nc, -1), pos(nc, -1), rowJ;
    std::vector<int> off1(1, 0), la, lp, cnt;
    for (int64_t i = 0; i < n; ++i) {
      rowJ.clear();
      for (int q = ar[i]; q < ar[i + 1]; ++q) {
        const int k = ac[q];
        for (int t = pr[k]; t < pr[k + 1]; ++t) {
          const int J = pc[t];
          if (mark[J] != (int)i) {
            mark[J] = (int)i;
            rowJ.push_back(J);
          }
        }
      }
      std::sort(rowJ.begin(), rowJ.end());
      const int z0 = (int)zc.size();
      for (size_t u = 0; u < rowJ.size(); ++u) {
        pos[rowJ[u]] = z0 + (int)u;
        zc.push_back(rowJ[u]);
      }
      zr[i + 1] = (int)zc.size();
      cnt.assign(rowJ.size(), 0);
      for (int q = ar[i]; q < ar[i + 1]; ++q)
        for (int t = pr[ac[q]]; t < pr[ac[q] + 1]; ++t) cnt[pos[pc[t]] - z0]++;
      const size_t base = la.size();
      std::vector<int> fill(rowJ.size());
      size_t acc = base;
      for (size_t u = 0; u < rowJ.size(); ++u) {
        fill[u] = (int)acc;
        acc += cnt[u];
        off1.push_back((int)acc);
      }
      la.resize(acc);
      lp.resize(acc);
      for (int q = ar[i]; q < ar[i + 1]; ++q) {
        const int k = ac[q];
        for (int t = pr[k]; t < pr[k + 1]; ++t) {
          const int u = pos[pc[t]] - z0;
          la[fill[u]] = aslot[q];
          lp[fill[u]] = t;
          fill[u]++;
        }
      }
      if (la.size() >= (size_t)INT32_MAX) return make_status(BAMG_ERR_INVALID, "Galerkin product too large");
    }
    pl->nz = (int64_t)zc.size();
    pl->n1 = pl->nz;
    pl->e1 = (int64_t)la.size();
    {
      pl->rounds1 = item_rounds(pl->n1, bsp, pl->ctx->sm_count);
      std::vector<int> order = order_by_work(off1, pl->rounds1 * 8 * (32 / bsp)), noff, na, np;
      permute_lists(order, off1, la, lp, noff, na, np);
      BAMG_TRY(upload(&pl->s1_z, order, st));
      BAMG_TRY(upload(&pl->s1_off, noff, st));
      BAMG_TRY(upload(&pl->s1_a, na, st));
      BAMG_TRY(upload(&pl->s1_p, np, st));
      BAMG_CUDA(cudaStreamSynchronize(st));
    }
    BAMG_TRY(dalloc(&pl->Z, pl->nz * bs * bsp, st));
    if (!want_ac) return Status{};

    // ---- A_c pattern and stage-2 lists: rows I over R_I = {(i, t): P(i, I) = t}
    std::vector<int> rr(nc + 1, 0), ri, rt;
    for (int64_t t = 0; t < (int64_t)pc.size(); ++t) rr[pc[t] + 1]++;
    for (int64_t I = 0; I < nc; ++I) rr[I + 1] += rr[I];
    ri.resize(pc.size());
    rt.resize(pc.size());
    {
      std::vector<int> fill(rr.begin(), rr.end() - 1);
      for (int64_t i = 0; i < n; ++i)
        for (int t = pr[i]; t < pr[i + 1]; ++t) {
          const int I = pc[t];
          ri[fill[I]] = (int)i;
          rt[fill[I]] = t;
          fill[I]++;
        }
    }
    std::vector<int> cr(nc + 1, 0), ccol;
    std::vector<int> off2, l2p, l2z, item_ac;
    std::fill(mark.begin(), mark.end(), -1);
    std::vector<std::vector<std::pair<int, int>>> rowlists;
    for (int64_t I = 0; I < nc; ++I) {
      rowJ.clear();
      for (int u = rr[I]; u < rr[I + 1]; ++u) {
        const int i = ri[u];
        for (int z = zr[i]; z < zr[i + 1]; ++z) {
          const int J = zc[z];
          if (mark[J] != (int)I) {
            mark[J] = (int)I;
            rowJ.push_back(J);
          }
        }
      }
      std::sort(rowJ.begin(), rowJ.end());
      const int c0 = (int)ccol.size();
      for (size_t u = 0; u < rowJ.size(); ++u) {
        pos[rowJ[u]] = (int)u;
        ccol.push_back(rowJ[u]);
      }
      cr[I + 1] = (int)ccol.size();
      rowlists.assign(rowJ.size(), {});
      for (int u = rr[I]; u < rr[I + 1]; ++u) {
        const int i = ri[u], t = rt[u];
        for (int z = zr[i]; z < zr[i + 1]; ++z) {
          const int J = zc[z];
          if (pl->symmetric && J < I) continue;
          rowlists[pos[J]].push_back({t, z});
        }
      }
      for (size_t u = 0; u < rowJ.size(); ++u) {
        if (pl->symmetric && rowJ[u] < I) continue;
        item_ac.push_back(c0 + (int)u);
        off2.push_back((int)l2p.size());
        for (auto& e : rowlists[u]) {
          l2p.push_back(e.first);
          l2z.push_back(e.second);
        }
      }
      if (l2p.size() >= (size_t)INT32_MAX) return make_status(BAMG_ERR_INVALID, "Galerkin product too large");
    }
    off2.push_back((int)l2p.size());
    bamg_bsr* Ac = nullptr;
    if (bamg_bsr_create(ctx, bsp, bsp, nc, nc, &Ac) != BAMG_OK) return make_status(BAMG_ERR_OOM, "create A_c");
    *Ac_out = Ac;
    pl->Ac = Ac;
    Ac->symmetric = pl->symmetric;
    std::vector<int> crow_copy = cr, ccol_copy = ccol;
    BAMG_TRY(bsr_set_pattern(Ac, std::move(crow_copy), std::move(ccol_copy), kSortAuto));
    pl->ac_pid = Ac->pattern_id;
    const auto& cslot = Ac->h_slot_of;
    const auto& crp = Ac->h_rowptr;
    const auto& ccl = Ac->h_colidx;
    std::vector<int> islot(item_ac.size()), itslot(item_ac.size(), -1);
    std::vector<int> Irow(ccl.size());
    for (int64_t I = 0; I < nc; ++I)
      for (int k = crp[I]; k < crp[I + 1]; ++k) Irow[k] = (int)I;
    for (size_t it = 0; it < item_ac.size(); ++it) {
      const int k = item_ac[it];
      islot[it] = cslot[k];
      const int I = Irow[k], J = ccl[k];
      if (pl->symmetric && J != I) {
        auto b = ccl.begin() + crp[J], e = ccl.begin() + crp[J + 1];
        auto f = std::lower_bound(b, e, I);
        if (f == e || *f != I) return make_status(BAMG_ERR_INVALID, "symmetric A_c pattern is not symmetric");
        itslot[it] = cslot[crp[J] + (int)(f - b)];
      }
    }
    pl->n2 = (int64_t)item_ac.size();
    pl->e2 = (int64_t)l2p.size();
    std::vector<int> order = order_by_work(off2, std::max<int64_t>(1, pl->n2)), noff, np, nz;
    permute_lists(order, off2, l2p, l2z, noff, np, nz);
    std::vector<int> os(order.size()), ots(order.size());
    for (size_t t = 0; t < order.size(); ++t) {
      os[t] = islot[order[t]];
      ots[t] = itslot[order[t]];
    }
    BAMG_TRY(upload(&pl->s2_slot, os, st));
    BAMG_TRY(upload(&pl->s2_tslot, ots, st));
    BAMG_TRY(upload(&pl->s2_off, noff, st));
    BAMG_TRY(upload(&pl->s2_p, np, st));
    BAMG_TRY(upload(&pl->s2_z, nz, st));
    BAMG_CUDA(cudaStreamSynchronize(st));
    return Status{};
  }();
  if (!s.ok()) {
    ptap_release(pl);
    if (Ac_out && *Ac_out) {
      bamg_bsr_destroy(*Ac_out);
      *Ac_out = nullptr;
    }
    delete pl;
    return s;
  }
  *plan_out = pl;
  return Status{};
}

template <typename T>
static Status run_stages(bamg_ptap* pl, const T* Avals, const T* Pblk, T* Z, T* Acvals, bool stage2) {
  cudaStream_t st = pl->ctx->stream;
  const uint4* Acut = (const uint4*)pl->Acut;
  const uint4* Pcut = (const uint4*)pl->Pcut;
  const int G = 32 / pl->bsp;
  auto blocks_for = [&](int64_t items, int rounds) {
    const int64_t per = (int64_t)rounds * 8 * G;
    return (unsigned)((items + per - 1) / per);
  };
  if (pl->n1 > 0) {
    const unsigned b = blocks_for(pl->n1, pl->rounds1);
    const int pm = prof_begin(pl->ctx, pl->prof_stage1, st);
    if (pl->bs == 3 && pl->bsp == 6)
      { k_ptap_stage1<3, 6, T><<<b, 256, 0, st>>>(pl->n1, pl->rounds1, pl->s1_z, pl->s1_off, pl->s1_a, pl->s1_p, Avals, Pblk, Acut, Z); BAMG_COUNT_LAUNCH; }
    else if (pl->bs == 6 && pl->bsp == 6)
      { k_ptap_stage1<6, 6, T><<<b, 256, 0, st>>>(pl->n1, pl->rounds1, pl->s1_z, pl->s1_off, pl->s1_a, pl->s1_p, Avals, Pblk, Acut, Z); BAMG_COUNT_LAUNCH; }
    else
      { k_ptap_stage1<3, 3, T><<<b, 256, 0, st>>>(pl->n1, pl->rounds1, pl->s1_z, pl->s1_off, pl->s1_a, pl->s1_p, Avals, Pblk, Acut, Z); BAMG_COUNT_LAUNCH; }
    prof_end(pl->ctx, pm, st);
    BAMG_CUDA(cudaGetLastError());
  }
  if (stage2 && pl->n2 > 0) {
    // The coarser the level, the fewer and the longer the lists: warps share
    // them until there are 16 per SM sub-partition (64^3, level 1: 3,601 items
    // are 91 CTAs and took 321 us; 12^3, level 0: 125 -> 23 us shared by eight).
    int S = 1;
    while (S < 8 && pl->n2 / G * S < pl->ctx->sm_count * 4 * 16) S *= 2;
    const int64_t per = (int64_t)(8 / S) * G;
    const unsigned b = (unsigned)((pl->n2 + per - 1) / per);
    const int pm = prof_begin(pl->ctx, pl->prof_stage2, st);
#define BAMG_STAGE2(A, B, N)                                                                                       \
  k_ptap_stage2<A, B, N, T><<<b, 256, 0, st>>>(pl->n2, pl->s2_slot, pl->s2_tslot, pl->s2_off, pl->s2_p, pl->s2_z, \
                                               Pblk, Pcut, Z, Acvals)
#define BAMG_STAGE2_S(A, B)           \
  switch (S) {                        \
    case 8: BAMG_STAGE2(A, B, 8); break; \
    case 4: BAMG_STAGE2(A, B, 4); break; \
    case 2: BAMG_STAGE2(A, B, 2); break; \
    default: BAMG_STAGE2(A, B, 1); break; \
  }
    if (pl->bs == 3 && pl->bsp == 6) {
      BAMG_STAGE2_S(3, 6)
    } else if (pl->bs == 6 && pl->bsp == 6) {
      BAMG_STAGE2_S(6, 6)
    } else {
      BAMG_STAGE2_S(3, 3)
    }
#undef BAMG_STAGE2_S
#undef BAMG_STAGE2
    BAMG_COUNT_LAUNCH;
    prof_end(pl->ctx, pm, st);
    BAMG_CUDA(cudaGetLastError());
  }
  return Status{};
}

// State gate (Sec. 3.5): the block-ordered copy of P is rebuilt only when P's
// version differs from the cached one.
static Status refresh_pblk(bamg_ptap* pl, bamg_bsr* P, bool fp32) {
  cudaStream_t st = pl->ctx->stream;
  const int64_t ne = P->nnzb * P->block_elems();
  if (pl->pblk_version != P->version) {
    if (P->vals64_stale) return make_status(BAMG_ERR_STATE, "P holds only FP32 values");
    if (!pl->Pblk) BAMG_TRY(dalloc(&pl->Pblk, ne, st));
    BAMG_TRY(launch_gather_blocks(P, P->vals, pl->Pblk, st));
    pl->pblk_version = P->version;
    pl->pblk_refreshes++;
  }
  if (fp32 && pl->pblk32_version != P->version) {
    const int n = (int)P->block_elems(), pitch = block_pitch<float>(n);
    if (!pl->Pblk32) BAMG_TRY(dalloc(&pl->Pblk32, P->nnzb * pitch, st));
    if (P->nnzb > 0) {
      k_pad_blocks<<<(unsigned)((P->nnzb * pitch + 255) / 256), 256, 0, st>>>(P->nnzb, n, pitch, pl->Pblk, pl->Pblk32);
      BAMG_COUNT_LAUNCH;
      BAMG_CUDA(cudaGetLastError());
    }
    pl->pblk32_version = P->version;
  }
  return Status{};
}

// Cut copy of P's blocks for the FP64 second stage, behind the same state gate.
static Status refresh_pcut(bamg_ptap* pl, const bamg_bsr* P) {
  cudaStream_t st = pl->ctx->stream;
  if (pl->pcut_version == P->version || P->nnzb == 0) return Status{};
  const int words = pl->bs == 6 ? PCut<6, 6>::kWords : pl->bsp == 6 ? PCut<3, 6>::kWords : PCut<3, 3>::kWords;
  if (!pl->Pcut) BAMG_TRY(dalloc(&pl->Pcut, P->nnzb * words * 4, st));
  const unsigned b = (unsigned)((P->nnzb + 63) / 64);
  uint4* out = (uint4*)pl->Pcut;
  if (pl->bs == 6)
    k_cut_transposed<6, 6><<<b, 64, 0, st>>>(P->nnzb, pl->Pblk, out);
  else if (pl->bsp == 6)
    k_cut_transposed<3, 6><<<b, 64, 0, st>>>(P->nnzb, pl->Pblk, out);
  else
    k_cut_transposed<3, 3><<<b, 64, 0, st>>>(P->nnzb, pl->Pblk, out);
  BAMG_COUNT_LAUNCH;
  BAMG_CUDA(cudaGetLastError());
  pl->pcut_version = P->version;
  return Status{};
}

// Cut copy of A's blocks for this product (their values are new every time).
static Status cut_operator(bamg_ptap* pl, const bamg_bsr* A) {
  cudaStream_t st = pl->ctx->stream;
  const int64_t n = A->nslots();
  if (n == 0) return Status{};
  const int words = pl->bs == 6 ? ACut<6>::kWords : ACut<3>::kWords;
  if (!pl->Acut) BAMG_TRY(dalloc(&pl->Acut, n * words * 4, st));
  const unsigned b = (unsigned)((n + 63) / 64);
  const int pm = prof_begin(pl->ctx, pl->prof_stage1, st, 0);
  if (pl->bs == 6)
    k_cut_slots<6><<<b, 64, 0, st>>>(n, A->vals, (uint4*)pl->Acut);
  else
    k_cut_slots<3><<<b, 64, 0, st>>>(n, A->vals, (uint4*)pl->Acut);
  BAMG_COUNT_LAUNCH;
  prof_end(pl->ctx, pm, st);
  BAMG_CUDA(cudaGetLastError());
  return Status{};
}

// FP32 copy of A's blocks for this product, padded.
static Status pad_operator(bamg_ptap* pl, const bamg_bsr* A, float* Apad) {
  cudaStream_t st = pl->ctx->stream;
  const int64_t n = A->nslots();
  if (n == 0) return Status{};
  const unsigned b = (unsigned)((n + 127) / 128);
  const int pm = prof_begin(pl->ctx, pl->prof_stage1, st, 0);
  if (pl->bs == 6)
    k_pad_slots<6><<<b, 128, 0, st>>>(n, A->vals32, (float4*)Apad);
  else
    k_pad_slots<3><<<b, 128, 0, st>>>(n, A->vals32, (float4*)Apad);
  BAMG_COUNT_LAUNCH;
  prof_end(pl->ctx, pm, st);
  BAMG_CUDA(cudaGetLastError());
  return Status{};
}

Status ptap_run(bamg_ptap* pl, bamg_bsr* A, bamg_bsr* P, bamg_bsr* Ac, bamg_prec prec, bool stage2) {
  if (A != pl->A || P != pl->P || (stage2 && Ac != pl->Ac) || A->pattern_id != pl->a_pid ||
      P->pattern_id != pl->p_pid || (stage2 && Ac->pattern_id != pl->ac_pid))
    return make_status(BAMG_ERR_STATE, "Galerkin plan used with matrices it was not built for");
  if (stage2 && !pl->Ac) return make_status(BAMG_ERR_STATE, "plan has no coarse stage");
  cudaStream_t st = pl->ctx->stream;
  if (prec == BAMG_FP64) {
    if (A->vals64_stale) return make_status(BAMG_ERR_STATE, "A holds only FP32 values; use BAMG_FP32");
    BAMG_TRY(refresh_pblk(pl, P, false));
    if (stage2) BAMG_TRY(refresh_pcut(pl, P));
    BAMG_TRY(cut_operator(pl, A));
    BAMG_TRY(run_stages<double>(pl, A->vals, pl->Pblk, pl->Z, stage2 ? Ac->vals : nullptr, stage2));
    if (stage2) {
      Ac->version++;
      Ac->vals64_stale = false;
    } else {
      ptap_trim(pl);  // prolongator smoothing: setup only
    }
  } else if (prec == BAMG_FP32) {
    BAMG_TRY(bsr_ensure_fp32(A));
    BAMG_TRY(refresh_pblk(pl, P, true));
    if (stage2 && !Ac->vals32) BAMG_TRY(dalloc(&Ac->vals32, Ac->nslots() * Ac->block_elems(), st));
    if (stage2 && Ac->vals32 && Ac->vals32_version == ~0ull)
      BAMG_CUDA(cudaMemsetAsync(Ac->vals32, 0, sizeof(float) * Ac->nslots() * Ac->block_elems(), st));
    // The FP64 intermediate's memory, scratch of the other precision, holds A's
    // padded copy where that fits (3x3 blocks), or else the FP32 intermediate;
    // the other one is allocated by the first FP32 product (47^3: with both
    // allocated that product took 1,190 us, so 1,035).
    const int64_t na = A->nslots() * block_pitch<float>(pl->bs * pl->bs), nz = pl->nz * pl->bs * pl->bsp;
    const bool pad_in_z = na <= 2 * nz;
    if (pad_in_z && !pl->Z32) BAMG_TRY(dalloc(&pl->Z32, nz, st));
    if (!pad_in_z && !pl->Apad) BAMG_TRY(dalloc(&pl->Apad, na, st));
    float* Apad = pad_in_z ? reinterpret_cast<float*>(pl->Z) : pl->Apad;
    float* Z32 = pad_in_z ? pl->Z32 : reinterpret_cast<float*>(pl->Z);
    BAMG_TRY(pad_operator(pl, A, Apad));
    BAMG_TRY(run_stages<float>(pl, Apad, pl->Pblk32, Z32, stage2 ? Ac->vals32 : nullptr, stage2));
    if (stage2) {
      Ac->version++;
      Ac->vals32_version = Ac->version;
      Ac->vals64_stale = true;
    }
  } else {
    return make_status(BAMG_ERR_INVALID, "bad precision");
  }
  return Status{};
}

}  // namespace bamg

using namespace bamg;

extern "C" {

bamg_status bamg_ptap_symbolic(bamg_bsr* A, bamg_bsr* P, bamg_ptap** plan, bamg_bsr** Ac) {
  if (!A || !P || !plan || !Ac) return BAMG_ERR_INVALID;
  Status s = ptap_build(A, P, true, plan, Ac);
  return s.ok() ? BAMG_OK : fail(A->ctx, s);
}

bamg_status bamg_ptap_numeric(bamg_ptap* plan, bamg_bsr* A, bamg_bsr* P, bamg_bsr* Ac) {
  if (!plan || !A || !P || !Ac) return BAMG_ERR_INVALID;
  Status s = ptap_run(plan, A, P, Ac, BAMG_FP64, true);
  return s.ok() ? BAMG_OK : fail(plan->ctx, s);
}

bamg_status bamg_ptap_numeric_prec(bamg_ptap* plan, bamg_bsr* A, bamg_bsr* P, bamg_bsr* Ac, bamg_prec prec) {
  if (!plan || !A || !P || !Ac) return BAMG_ERR_INVALID;
  Status s = ptap_run(plan, A, P, Ac, prec, true);
  return s.ok() ? BAMG_OK : fail(plan->ctx, s);
}

bamg_status bamg_ptap_get_refreshes(const bamg_ptap* plan, uint64_t* p_refreshes) {
  if (!plan || !p_refreshes) return BAMG_ERR_INVALID;
  *p_refreshes = plan->pblk_refreshes;
  return BAMG_OK;
}

bamg_status bamg_ptap_destroy(bamg_ptap* plan) {
  if (!plan) return BAMG_OK;
  ptap_release(plan);
  delete plan;
  return BAMG_OK;
}

}  // extern "C"

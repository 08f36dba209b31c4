// Float contraction on the CUDA cores for the float configurations (and the bf16-storage networks that have no
// tensor-core kernels):   C(m, n) = sum_k A(m, k) * B(n, k),  k in the split's range, every output one chain of fused
// multiply-adds in ascending k (the forward pass keeps the order of its additions whatever the tile: a sum in another
// order puts units within rounding of zero on the other side of the ReLU).
//
// Operands are functors that give the address of 16 bytes of neighbouring values, in one of two orders:
//   K_CONTIG   (convolution windows, weights of the forward pass)  Row row(r);  const T* at(Row, k): k, k + 1, ... of row r
//   otherwise  (weight gradients, transposed weights)              Row row(r);  const T* at(Row, k): rows r, r + 1, ... at k
// or nullptr for zeros.  Row is worked out once per thread (a thread keeps its rows over all k blocks), so that the window's
// divisions are not paid per element.  Both orders lie in shared memory as they come, [row][k] or [k][row], so float
// operands are copied asynchronously, FF_STAGES - 1 blocks ahead; bytes and bf16 pass through registers to be widened.
//
// What bounds it: shared-memory reads into registers (128 bytes per clock and SM) against 128 multiply-adds per clock.  A lane
// with 8 x 8 outputs reads four k of eight rows and eight columns, sixteen 16-byte reads for 256 multiply-adds: one byte each,
// just what the pipe takes; 8 x 4 outputs take one and a half.  Problems with enough outputs therefore use 8 x 8 per lane;
// smaller ones, where latency counts, 4 x 4 or 2 x 4, so that more warps share the work (ff_shape in net_simt.cu picks).
// With 8 x 8 the issue slots then come first: 82 % of them busy, shared memory 46 % of the cycles, 20 of 36 TMAC/s (the larger
// network's fully connected weight gradient over 640 rows).
#pragma once
#include "common.cuh"

namespace paac {

// k per split for a requested number of splits, and how many splits that gives
inline int gemm_k_per_split(int K, int splits, int granule = 16) {
  const int kps = (K + splits - 1) / splits;
  return (kps + granule - 1) / granule * granule;
}
inline int gemm_k_splits(int K, int splits, int granule = 16) { const int kps = gemm_k_per_split(K, splits, granule); return (K + kps - 1) / kps; }

// sixteen bytes of stored values as floats
__device__ __forceinline__ void widen(const uint4 v, const float*, float4 (&f)[1]) {
  f[0] = make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w));
}
__device__ __forceinline__ void widen(const uint4 v, const bf16*, float4 (&f)[2]) {
  f[0] = widen4(make_uint2(v.x, v.y)); f[1] = widen4(make_uint2(v.z, v.w));
}
__device__ __forceinline__ void widen(const uint4 v, const uint8_t*, float4 (&f)[4]) {
  f[0] = widen4(v.x); f[1] = widen4(v.y); f[2] = widen4(v.z); f[3] = widen4(v.w);
}

// A k block of R rows in shared memory: [R][BK + 4] or [BK][R + 4] (the padding keeps the reads below free of conflicts).
template <class OP, int R, int BK> struct FfTile {
  static constexpr int LD = (OP::K_CONTIG ? BK : R) + 4, FLOATS = (OP::K_CONTIG ? R : BK) * LD;
};
// What one thread brings of a tile per k block.  (Plain loads, not the read-only path: the kernel may start while the one
// that writes its operands drains.)
template <class OP, int R, int BK, int NT> struct FfLoader {
  typedef typename OP::Elem T;
  typedef FfTile<OP, R, BK> Tile;
  static constexpr bool ASYNC = sizeof(T) == 4;
  static constexpr int V = 16 / (int)sizeof(T), ROW_ITEMS = (OP::K_CONTIG ? BK : R) / V;
  static constexpr int ITEMS = R * BK / V, PER = (ITEMS + NT - 1) / NT;
  static constexpr bool FULL = ITEMS % NT == 0;
  typename OP::Row row[PER];
  uint4 val[ASYNC ? 1 : PER];
  __device__ __forceinline__ static int row_of(int i) { return OP::K_CONTIG ? i / ROW_ITEMS : (i % ROW_ITEMS) * V; }
  __device__ __forceinline__ static int k_of(int i) { return OP::K_CONTIG ? (i % ROW_ITEMS) * V : i / ROW_ITEMS; }
  __device__ __forceinline__ void init(const OP& op, int r0, int rows) {
#pragma unroll
    for (int it = 0; it < PER; ++it) {
      const int r = r0 + row_of(threadIdx.x + it * NT);
      row[it] = op.row(r < rows ? r : -1);
    }
  }
  // asks for a block: straight into shared memory, or into registers
  __device__ __forceinline__ void fetch(const OP& op, int k0, int k_end, float* tile) {
#pragma unroll
    for (int it = 0; it < PER; ++it) {
      const int i = threadIdx.x + it * NT;
      if (!FULL && i >= ITEMS) break;
      const int k = k0 + k_of(i);
      const T* src = k < k_end ? op.at(row[it], k) : nullptr;
      if constexpr (ASYNC) {
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(tile + (OP::K_CONTIG ? row_of(i) * Tile::LD + k_of(i) : k_of(i) * Tile::LD + row_of(i)));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src ? src : reinterpret_cast<const T*>(op.any())), "r"(src ? 16 : 0) : "memory");
      } else {
        val[it] = src ? *reinterpret_cast<const uint4*>(src) : make_uint4(0u, 0u, 0u, 0u);
      }
    }
  }
  // from registers to shared memory
  __device__ __forceinline__ void store(float* tile) const {
    if constexpr (!ASYNC) {
#pragma unroll
      for (int it = 0; it < PER; ++it) {
        const int i = threadIdx.x + it * NT;
        if (!FULL && i >= ITEMS) break;
        float4 f[V / 4];
        float4* dst = reinterpret_cast<float4*>(tile + (OP::K_CONTIG ? row_of(i) * Tile::LD + k_of(i) : k_of(i) * Tile::LD + row_of(i)));
        if constexpr (sizeof(T) == 1 && !OP::K_CONTIG) {
          // neighbouring threads' pieces are 64 bytes apart: each begins with another quarter of its own, so that eight threads'
          // stores lie in different banks (a quarter of the first layer's weight gradient's shared-memory cycles were such conflicts)
          const uint32_t turn = threadIdx.x >> 1;
          const uint4 v = val[it];
          const uint4 a = turn & 1u ? make_uint4(v.y, v.z, v.w, v.x) : v;
          widen(turn & 2u ? make_uint4(a.z, a.w, a.x, a.y) : a, (const T*)nullptr, f);
#pragma unroll
          for (int q = 0; q < V / 4; ++q) dst[(q + turn) & 3u] = f[q];
        } else {
          widen(val[it], (const T*)nullptr, f);
#pragma unroll
          for (int q = 0; q < V / 4; ++q) dst[q] = f[q];
        }
      }
    }
  }
};
// four k of a lane's T rows: f[k][row]; the lane's rows are lane, lane + LANES, ... (K_CONTIG) or runs of four (two for T = 2)
template <class OP, int R, int BK, int T, int LANES> __device__ __forceinline__ void ff_fragment(const float* tile, int row0, int lane, int k, float (&f)[4][T]) {
  constexpr int LD = FfTile<OP, R, BK>::LD;
  if constexpr (OP::K_CONTIG) {
#pragma unroll
    for (int i = 0; i < T; ++i) {
      const float4 v = *reinterpret_cast<const float4*>(tile + (row0 + lane + i * LANES) * LD + k);
      f[0][i] = v.x; f[1][i] = v.y; f[2][i] = v.z; f[3][i] = v.w;
    }
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if constexpr (T == 2) {
        const float2 v = *reinterpret_cast<const float2*>(tile + (k + q) * LD + row0 + lane * 2);
        f[q][0] = v.x; f[q][1] = v.y;
      } else {
#pragma unroll
        for (int g = 0; g < T / 4; ++g) {
          const float4 v = *reinterpret_cast<const float4*>(tile + (k + q) * LD + row0 + (g * LANES + lane) * 4);
          f[q][4 * g] = v.x; f[q][4 * g + 1] = v.y; f[q][4 * g + 2] = v.z; f[q][4 * g + 3] = v.w;
        }
      }
    }
  }
}
// which row (of the warp's) fragment element i of a lane is
template <bool K_CONTIG, int T, int LANES> __device__ __forceinline__ int ff_index(int lane, int i) {
  constexpr int RUN = T < 4 ? T : 4;
  return K_CONTIG ? lane + i * LANES : ((i / RUN) * LANES + lane) * RUN + i % RUN;
}

// WM x WN warps; a warp's lanes are LM x (32 / LM), TM x TN outputs each.  Grid (m tiles, n tiles, splits x classes).
// With EP::COLSUM the epilogue also gets the sum over k of every row of B (bias gradients), once per split.
constexpr int FF_STAGES = 3;
template <int LM, int TM, int TN, int WM, int WN, int BK, class LA, class LB> struct FfCfg {
  static constexpr int LN = 32 / LM, BM = LM * TM * WM, BN = LN * TN * WN, NT = 32 * WM * WN;
  static constexpr int A_FLOATS = FfTile<LA, BM, BK>::FLOATS, STAGE = A_FLOATS + FfTile<LB, BN, BK>::FLOATS;
  static constexpr int SMEM = FF_STAGES * STAGE * 4;
};
template <int LM, int TM, int TN, int WM, int WN, int BK, class LA, class LB, class EP>
__global__ void __launch_bounds__(32 * WM * WN, 12 / (WM * WN))
gemm_ffma_kernel(int M, int N, int K, int k_per_split, int splits, LA la, LB lb, EP ep) {
  pdl_entry();
  typedef FfCfg<LM, TM, TN, WM, WN, BK, LA, LB> C;
  constexpr int LN = C::LN, BM = C::BM, BN = C::BN, NT = C::NT;
  extern __shared__ __align__(16) float ff_smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int lx = lane % LN, ly = lane / LN, wm = warp % WM, wn = warp / WM;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  const int split = blockIdx.z % splits, cls = blockIdx.z / splits;
  la.enter(cls); lb.enter(cls); ep.enter(cls);
  const int k_begin = split * k_per_split, k_end = min(K, k_begin + k_per_split);

  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
  FfLoader<LA, BM, BK, NT> fa;
  FfLoader<LB, BN, BK, NT> fb;
  float colsum = 0.f;              // thread n < BN of the first tile row: the sum over k of column n, in order
  fa.init(la, m0, M);
  fb.init(lb, n0, N);
  auto stage_of = [&](int block) { return ff_smem + (block % FF_STAGES) * C::STAGE; };
  // operands that pass through registers are one block ahead, asynchronous ones FF_STAGES - 1
  const int blocks = k_end > k_begin ? (k_end - k_begin + BK - 1) / BK : 0;
#pragma unroll
  for (int q = 0; q < FF_STAGES - 1; ++q) {
    if (q < blocks) {
      if (fa.ASYNC || q == 0) fa.fetch(la, k_begin + q * BK, k_end, stage_of(q));
      if (fb.ASYNC || q == 0) fb.fetch(lb, k_begin + q * BK, k_end, stage_of(q) + C::A_FLOATS);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  if (blocks > 0) { fa.store(stage_of(0)); fb.store(stage_of(0) + C::A_FLOATS); }
  for (int i = 0; i < blocks; ++i) {
    asm volatile("cp.async.wait_group %0;" ::"n"(FF_STAGES - 2) : "memory");
    __syncthreads();               // block i is in; everyone is done with the stage of block i - 1
    const int ahead = i + FF_STAGES - 1;
    if (fa.ASYNC && ahead < blocks) fa.fetch(la, k_begin + ahead * BK, k_end, stage_of(ahead));
    if (fb.ASYNC && ahead < blocks) fb.fetch(lb, k_begin + ahead * BK, k_end, stage_of(ahead) + C::A_FLOATS);
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (!fa.ASYNC && i + 1 < blocks) fa.fetch(la, k_begin + (i + 1) * BK, k_end, nullptr);
    if (!fb.ASYNC && i + 1 < blocks) fb.fetch(lb, k_begin + (i + 1) * BK, k_end, nullptr);
    const float* ta = stage_of(i);
    const float* tb = ta + C::A_FLOATS;
#pragma unroll
    for (int k = 0; k < BK; k += 4) {
      float a[4][TM], b[4][TN];
      ff_fragment<LA, BM, BK, TM, LM>(ta, wm * LM * TM, ly, k, a);
      ff_fragment<LB, BN, BK, TN, LN>(tb, wn * LN * TN, lx, k, b);
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int x = 0; x < TM; ++x)
#pragma unroll
          for (int y = 0; y < TN; ++y) acc[x][y] = fmaf(a[q][x], b[q][y], acc[x][y]);
    }
    if constexpr (EP::COLSUM) {
      static_assert(!LB::K_CONTIG && BN <= NT, "weight gradients");
      if (blockIdx.x == 0 && threadIdx.x < BN)
#pragma unroll
        for (int k = 0; k < BK; ++k) colsum += tb[k * FfTile<LB, BN, BK>::LD + threadIdx.x];
    }
    if (!fa.ASYNC && i + 1 < blocks) fa.store(stage_of(i + 1));
    if (!fb.ASYNC && i + 1 < blocks) fb.store(stage_of(i + 1) + C::A_FLOATS);
  }
#pragma unroll
  for (int x = 0; x < TM; ++x) {
    const int m = m0 + wm * LM * TM + ff_index<LA::K_CONTIG, TM, LM>(ly, x);
    if (m >= M) continue;
    if constexpr (LB::K_CONTIG) {
#pragma unroll
      for (int y = 0; y < TN; ++y) {
        const int n = n0 + wn * LN * TN + ff_index<true, TN, LN>(lx, y);
        if (n < N) ep(m, n, acc[x][y], split);
      }
    } else {
#pragma unroll
      for (int y = 0; y < TN; y += 4) {
        const int n = n0 + wn * LN * TN + ff_index<false, TN, LN>(lx, y);
        if (n < N) ep(m, n, make_float4(acc[x][y], acc[x][y + 1], acc[x][y + 2], acc[x][y + 3]), split);
      }
    }
  }
  if constexpr (EP::COLSUM) {
    if (blockIdx.x == 0 && threadIdx.x < BN && n0 + threadIdx.x < N) ep.colsum(n0 + threadIdx.x, colsum, split);
  }
}

template <int LM, int TM, int TN, int WM, int WN, int BK, class LA, class LB, class EP>
inline void gemm_ffma(LaunchCtx& lc, int kid, int M, int N, int K, int k_per_split, int classes, LA la, LB lb, EP ep) {
  typedef FfCfg<LM, TM, TN, WM, WN, BK, LA, LB> C;
  auto kern = gemm_ffma_kernel<LM, TM, TN, WM, WN, BK, LA, LB, EP>;
  static const cudaError_t attr = C::SMEM > 48 * 1024 ? cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM) : cudaSuccess;
  if (attr != cudaSuccess) lc.host_failure = true;
  const int splits = (K + k_per_split - 1) / k_per_split;
  KernelScope scope(lc, kid);
  launch_kernel_overlapped(lc, kern, dim3((M + C::BM - 1) / C::BM, (N + C::BN - 1) / C::BN, splits * classes), dim3(C::NT), C::SMEM, M, N, K,
                           k_per_split, splits, la, lb, ep);
}

// ---- operands ------------------------------------------------------------------------------------------------------
// (enter(c): class c of a launch that runs several contractions side by side)
// x[row][k], rows ld apart
template <class T> struct FfRows {
  static constexpr bool K_CONTIG = true;
  typedef T Elem;
  typedef const T* Row;
  const T* p; int ld;
  __device__ __forceinline__ const T* any() const { return p; }
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ Row row(int r) const { return r >= 0 ? p + (size_t)r * ld : nullptr; }
  __device__ __forceinline__ const T* at(Row b, int k) const { return b ? b + k : nullptr; }
};
// x[k][row]
template <class T> struct FfCols {
  static constexpr bool K_CONTIG = false;
  typedef T Elem;
  typedef const T* Row;
  const T* p; int ld;
  __device__ __forceinline__ const T* any() const { return p; }
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ Row row(int r) const { return r >= 0 ? p + r : nullptr; }
  __device__ __forceinline__ const T* at(Row b, int k) const { return b ? b + (size_t)k * ld : nullptr; }
};
// convolution window: row = (state, oh, ow), k = (r, s, ci); the K C values of a filter row are contiguous
template <class G, class T> struct FfWindow {
  static constexpr bool K_CONTIG = true;
  typedef T Elem;
  typedef const T* Row;
  const T* x;
  __device__ __forceinline__ const T* any() const { return x; }
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ Row row(int m) const {
    if (m < 0) return nullptr;
    const int b = m / (G::OH * G::OW), rem = m % (G::OH * G::OW), oh = rem / G::OW, ow = rem % G::OW;
    return x + ((size_t)(b * G::H + oh * G::S) * G::W + ow * G::S) * G::C;
  }
  __device__ __forceinline__ const T* at(Row b, int k) const {
    return b ? b + (k / (G::K * G::C)) * (G::W * G::C) + k % (G::K * G::C) : nullptr;
  }
};
// the same window from the weight gradient: row j = (r, s, ci), k = (state, oh, ow)
template <class G, class T> struct FfWindowT {
  static constexpr bool K_CONTIG = false;
  typedef T Elem;
  typedef const T* Row;
  const T* x;
  __device__ __forceinline__ const T* any() const { return x; }
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ Row row(int j) const { return j >= 0 ? x + (j / (G::K * G::C)) * (G::W * G::C) + j % (G::K * G::C) : nullptr; }
  __device__ __forceinline__ const T* at(Row base, int m) const {
    if (!base) return nullptr;
    const int b = m / (G::OH * G::OW), rem = m % (G::OH * G::OW), oh = rem / G::OW, ow = rem % G::OW;
    return base + ((size_t)(b * G::H + oh * G::S) * G::W + ow * G::S) * G::C;
  }
};
// data gradient of a stride-1 layer: row = (state, y, x) of the layer input, k = (r, s, co); zero outside the output map
template <class G, class T> struct FfDgradWindow {
  static constexpr bool K_CONTIG = true;
  typedef T Elem;
  struct Row { const T* b; int y, x; };
  const T* g;
  __device__ __forceinline__ const T* any() const { return g; }
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ Row row(int m) const {
    if (m < 0) return Row{nullptr, 0, 0};
    const int b = m / (G::H * G::W), rem = m % (G::H * G::W);
    return Row{g + (size_t)b * G::OH * G::OW * G::CO, rem / G::W, rem % G::W};
  }
  __device__ __forceinline__ const T* at(const Row& q, int k) const {
    const int tap = k / G::CO, oh = q.y - tap / G::K, ow = q.x - tap % G::K;
    if (!q.b || (unsigned)oh >= (unsigned)G::OH || (unsigned)ow >= (unsigned)G::OW) return nullptr;
    return q.b + (oh * G::OW + ow) * G::CO + k % G::CO;
  }
};
template <class G, class T> struct FfWeightT {              // row = ci, k = (r, s, co)
  static constexpr bool K_CONTIG = false;
  typedef T Elem;
  typedef const T* Row;
  const T* w;
  __device__ __forceinline__ const T* any() const { return w; }
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ Row row(int r) const { return r >= 0 ? w + r : nullptr; }
  __device__ __forceinline__ const T* at(Row b, int k) const {
    return b ? b + ((k % G::CO) * (G::K * G::K) + k / G::CO) * G::C : nullptr;
  }
};
// Stride 2, 4 x 4 kernel: the input pixels of parity class (py, px) are touched by the four taps (py + 2 i, px + 2 j)
// only, a dense contraction of its own with a quarter of the reduction.  Row = (state, y >> 1, x >> 1), k = (i, j, co).
template <class G, class T> struct FfDgradClass {
  static constexpr bool K_CONTIG = true;
  typedef T Elem;
  struct Row { const T* b; int y, x; };
  const T* g;
  __device__ __forceinline__ const T* any() const { return g; }
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ Row row(int m) const {
    constexpr int HH = G::H / 2, WW = G::W / 2;
    if (m < 0) return Row{nullptr, 0, 0};
    const int b = m / (HH * WW), rem = m % (HH * WW);
    return Row{g + (size_t)b * G::OH * G::OW * G::CO, rem / WW, rem % WW};
  }
  __device__ __forceinline__ const T* at(const Row& q, int k) const {
    const int tap = k / G::CO, oh = q.y - (tap >> 1), ow = q.x - (tap & 1);
    if (!q.b || (unsigned)oh >= (unsigned)G::OH || (unsigned)ow >= (unsigned)G::OW) return nullptr;
    return q.b + (oh * G::OW + ow) * G::CO + k % G::CO;
  }
};
template <class G, class T> struct FfWeightClass {          // row = ci, k = (i, j, co) -> tap (py + 2 i, px + 2 j)
  static constexpr bool K_CONTIG = false;
  typedef T Elem;
  typedef const T* Row;
  const T* w; int z;
  __device__ __forceinline__ const T* any() const { return w; }
  __device__ __forceinline__ void enter(int c) { z = c; }
  __device__ __forceinline__ Row row(int r) const { return r >= 0 ? w + r + ((z >> 1) * G::K + (z & 1)) * G::C : nullptr; }
  __device__ __forceinline__ const T* at(Row b, int k) const {
    const int tap = k / G::CO;
    return b ? b + (((k % G::CO) * G::K + 2 * (tap >> 1)) * G::K + 2 * (tap & 1)) * G::C : nullptr;
  }
};

// ---- results -------------------------------------------------------------------------------------------------------
template <class T> struct FfBiasRelu {                       // out[m][n] = relu(acc * scale + bias[n])
  static constexpr bool COLSUM = false;
  T* out; const float* bias; int ld; float scale;
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ void operator()(int m, int n, float v, int) const {
    out[(size_t)m * ld + n] = from_f<T>(fmaxf(fmaf(v, scale, bias[n]), 0.f));
  }
  __device__ __forceinline__ void operator()(int m, int n, float4 v, int) const {
    store4(out + (size_t)m * ld + n, make_float4(fmaxf(fmaf(v.x, scale, bias[n]), 0.f), fmaxf(fmaf(v.y, scale, bias[n + 1]), 0.f),
                                                 fmaxf(fmaf(v.z, scale, bias[n + 2]), 0.f), fmaxf(fmaf(v.w, scale, bias[n + 3]), 0.f)));
  }
};
template <class T> struct FfReluMask {                       // out[m][n] = act[m][n] > 0 ? acc : 0
  static constexpr bool COLSUM = false;
  T* out; const T* act; int ld;
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ void operator()(int m, int n, float4 v, int) const {
    const size_t i = (size_t)m * ld + n;
    const float4 on = load4(act + i);
    store4(out + i, make_float4(on.x > 0.f ? v.x : 0.f, on.y > 0.f ? v.y : 0.f, on.z > 0.f ? v.z : 0.f, on.w > 0.f ? v.w : 0.f));
  }
};
template <class G, class T> struct FfReluMaskClass {         // the same for parity class z: row (state, y >> 1, x >> 1)
  static constexpr bool COLSUM = false;
  T* out; const T* act; int z;
  __device__ __forceinline__ void enter(int c) { z = c; }
  __device__ __forceinline__ void operator()(int m, int n, float4 v, int) const {
    constexpr int HH = G::H / 2, WW = G::W / 2;
    const int s = m / (HH * WW), rem = m % (HH * WW), y = 2 * (rem / WW) + (z >> 1), x = 2 * (rem % WW) + (z & 1);
    const size_t i = ((size_t)(s * G::H + y) * G::W + x) * G::C + n;
    const float4 on = load4(act + i);
    store4(out + i, make_float4(on.x > 0.f ? v.x : 0.f, on.y > 0.f ? v.y : 0.f, on.z > 0.f ? v.z : 0.f, on.w > 0.f ? v.w : 0.f));
  }
};
struct FfPartial {                                           // part[split][m][n]
  static constexpr bool COLSUM = false;
  float* part; int M, N;
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ void operator()(int m, int n, float v, int split) const { part[((size_t)split * M + m) * N + n] = v; }
  __device__ __forceinline__ void operator()(int m, int n, float4 v, int split) const {
    store4(part + ((size_t)split * M + m) * N + n, v);
  }
};
struct FfPartialColsum : FfPartial {                         // and the sum over k of B's rows: colpart[split][n]
  static constexpr bool COLSUM = true;
  float* colpart;
  __device__ __forceinline__ void colsum(int n, float v, int split) const { colpart[(size_t)split * N + n] = v; }
};

}  // namespace paac

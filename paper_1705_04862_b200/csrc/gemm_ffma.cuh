// Float contraction on the CUDA cores for the float configurations (and the bf16-storage networks that have no
// tensor-core kernels):   C(m, n) = sum_k A(m, k) * B(n, k),  k in the split's range.
//
// Operands are functors that hand out four neighbouring values with one load, in one of two orders:
//   K_CONTIG   (convolution windows, weights of the forward pass)  Row row(r);  float4 load(Row, k): k .. k + 3 of row r
//   otherwise  (weight gradients, transposed weights)              Row row(r);  float4 load(Row, k): rows r .. r + 3 at k
// Row is worked out once per thread (a thread keeps its rows over all k blocks), so that the window's divisions are not
// paid per element.
//
// What bounds it: the FMA pipe, and before that the issue slots.  The multiply-adds are fma.rn.f32x2, two per
// instruction: the two halves of an accumulator register pair are the sums over the even and over the odd k, so both
// operands come straight out of shared memory as (k, k + 1) pairs (no duplication of either) and the halves are added
// once, in the epilogue.  A warp owns 32 x 8 TN outputs (8 x TN per lane, lanes 4 x 8); its three (five for TN = 2)
// 16-byte reads per k pair are free of bank conflicts.  WM x WN warps cover the tile; with KG > 1 the warps come in KG
// groups that take alternating slices of every k block and are added, in order, through shared memory at the end:
// for problems with too few tiles to give every scheduler a warp.
#pragma once
#include "common.cuh"

namespace paac {

typedef unsigned long long f32x2;     // two floats, (low, high) = (even k, odd k)
__device__ __forceinline__ void fma2(f32x2& d, f32x2 a, f32x2 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b)); }
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float halves_sum(f32x2 v) {
  float lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
  return lo + hi;
}

// Four neighbouring stored values as floats.  Plain loads, not the read-only path: a kernel of this file may start while
// the one that writes its operands drains.
__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4(const bf16* p) {
  const uint2 v = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xFFFF0000u), __uint_as_float(v.y << 16),
                     __uint_as_float(v.y & 0xFFFF0000u));
}
// a byte in the low mantissa bits of 2^23 is 2^23 + byte: two full-rate instructions instead of a conversion
__device__ __forceinline__ float4 load4(const uint8_t* p) {
  const uint32_t v = *reinterpret_cast<const uint32_t*>(p);
  constexpr float BIAS = 8388608.f;
  return make_float4(__uint_as_float(__byte_perm(v, 0x4B000000u, 0x7440)) - BIAS, __uint_as_float(__byte_perm(v, 0x4B000000u, 0x7441)) - BIAS,
                     __uint_as_float(__byte_perm(v, 0x4B000000u, 0x7442)) - BIAS, __uint_as_float(__byte_perm(v, 0x4B000000u, 0x7443)) - BIAS);
}
__device__ __forceinline__ void store2(float* p, float a, float b) { *reinterpret_cast<float2*>(p) = make_float2(a, b); }
__device__ __forceinline__ void store2(bf16* p, float a, float b) { *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(a, b); }

template <int R, int BK> struct FfTile {              // R rows of a k block as (k, k + 1) pairs
  static constexpr int LD = R + 2;                    // 16-byte aligned; the two padding pairs spread the k rows over the banks
  float2 v[BK / 2][LD];
};
// what one thread fetches of a tile per k block
template <class OP, int R, int BK, int NT> struct FfLoader {
  static constexpr int ITEMS = OP::K_CONTIG ? R * BK / 4 : (R / 4) * (BK / 2);
  static constexpr int PER = (ITEMS + NT - 1) / NT;
  static constexpr bool FULL = ITEMS % NT == 0;
  typename OP::Row row[PER];
  float4 val[PER][OP::K_CONTIG ? 1 : 2];
  __device__ __forceinline__ void init(const OP& op, int r0, int rows) {
#pragma unroll
    for (int it = 0; it < PER; ++it) {
      const int i = threadIdx.x + it * NT;
      const int r = r0 + (OP::K_CONTIG ? i / (BK / 4) : (i % (R / 4)) * 4);
      row[it] = op.row(r < rows ? r : -1);
    }
  }
  __device__ __forceinline__ void fetch(const OP& op, int k0, int k_end) {
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int it = 0; it < PER; ++it) {
      const int i = threadIdx.x + it * NT;
      if (!FULL && i >= ITEMS) break;
      if constexpr (OP::K_CONTIG) {
        const int k = k0 + (i % (BK / 4)) * 4;
        val[it][0] = k < k_end ? op.load(row[it], k) : zero;
      } else {
        const int k = k0 + (i / (R / 4)) * 2;
        val[it][0] = k < k_end ? op.load(row[it], k) : zero;
        val[it][1] = k + 1 < k_end ? op.load(row[it], k + 1) : zero;
      }
    }
  }
  __device__ __forceinline__ void add_to(float4 (&sum)[PER]) const {          // a float4 of rows at two k
#pragma unroll
    for (int it = 0; it < PER; ++it) {
      if (!FULL && (int)threadIdx.x + it * NT >= ITEMS) break;
      sum[it].x += val[it][0].x + val[it][1].x; sum[it].y += val[it][0].y + val[it][1].y;
      sum[it].z += val[it][0].z + val[it][1].z; sum[it].w += val[it][0].w + val[it][1].w;
    }
  }
  __device__ __forceinline__ void store(FfTile<R, BK>& t) const {
#pragma unroll
    for (int it = 0; it < PER; ++it) {
      const int i = threadIdx.x + it * NT;
      if (!FULL && i >= ITEMS) break;
      if constexpr (OP::K_CONTIG) {
        const int kp = (i % (BK / 4)) * 2, r = i / (BK / 4);
        t.v[kp][r] = make_float2(val[it][0].x, val[it][0].y);
        t.v[kp + 1][r] = make_float2(val[it][0].z, val[it][0].w);
      } else {
        const int kp = i / (R / 4), r = (i % (R / 4)) * 4;
        float4* dst = reinterpret_cast<float4*>(&t.v[kp][r]);
        dst[0] = make_float4(val[it][0].x, val[it][1].x, val[it][0].y, val[it][1].y);
        dst[1] = make_float4(val[it][0].z, val[it][1].z, val[it][0].w, val[it][1].w);
      }
    }
  }
};

// grid (m tiles, n tiles, splits x classes).  The epilogue gets two neighbouring columns at a time; with EP::COLSUM also
// the sum over k of every row of B (bias gradients), once per split.
template <int WM, int WN, int TN, int KG, class LA, class LB, class EP>
__global__ void __launch_bounds__(32 * WM * WN * KG, WM * WN * KG == 4 ? 3 : 1)
gemm_ffma_kernel(int M, int N, int K, int k_per_split, int splits, LA la, LB lb, EP ep) {
  pdl_entry();
  constexpr int TM = 8, WTN = 8 * TN, BM = 32 * WM, BN = WTN * WN, BK = 16 * KG, NT = 32 * WM * WN * KG;
  constexpr int STAGES = 2 * (sizeof(FfTile<BM, BK>) + sizeof(FfTile<BN, BK>)) <= 48 * 1024 ? 2 : 1;
  __shared__ __align__(16) FfTile<BM, BK> As[STAGES];
  __shared__ __align__(16) FfTile<BN, BK> Bs[STAGES];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tx = lane & 7, ty = lane >> 3;
  const int wm = warp % WM, wn = (warp / WM) % WN, kg = warp / (WM * WN);
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  const int split = blockIdx.z % splits, cls = blockIdx.z / splits;
  la.enter(cls); lb.enter(cls); ep.enter(cls);
  const int k_begin = split * k_per_split, k_end = min(K, k_begin + k_per_split);

  f32x2 acc[TM][TN];
#pragma unroll
  for (int j = 0; j < TN; ++j)
#pragma unroll
    for (int i = 0; i < TM; ++i) acc[i][j] = 0ull;
  FfLoader<LA, BM, BK, NT> fa;
  FfLoader<LB, BN, BK, NT> fb;
  float4 colsum[EP::COLSUM ? FfLoader<LB, BN, BK, NT>::PER : 1];      // this thread's share of the sums over k of B's rows
#pragma unroll
  for (auto& c : colsum) c = make_float4(0.f, 0.f, 0.f, 0.f);
  fa.init(la, m0, M);
  fb.init(lb, n0, N);
  fa.fetch(la, k_begin, k_end); fb.fetch(lb, k_begin, k_end);
  int s = 0;
  for (int k0 = k_begin; k0 < k_end; k0 += BK, s ^= STAGES - 1) {
    // with two stages the barrier below also says that everyone is done with the stage written two blocks ago
    if (STAGES == 1 && k0 > k_begin) __syncthreads();
    fa.store(As[s]); fb.store(Bs[s]);
    if constexpr (EP::COLSUM) { if (blockIdx.x == 0) fb.add_to(colsum); }
    __syncthreads();
    if (k0 + BK < k_end) { fa.fetch(la, k0 + BK, k_end); fb.fetch(lb, k0 + BK, k_end); }
    const float2* pa = &As[s].v[kg * 8][wm * 32 + ty * 2];
    const float2* pb = &Bs[s].v[kg * 8][wn * WTN + tx * 2];
#pragma unroll
    for (int kp = 0; kp < 8; ++kp) {
      f32x2 a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; i += 2) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(pa + kp * FfTile<BM, BK>::LD + i * 4);
        a[i] = v.x; a[i + 1] = v.y;
      }
#pragma unroll
      for (int j = 0; j < TN; j += 2) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(pb + kp * FfTile<BN, BK>::LD + j * 8);
        b[j] = v.x; b[j + 1] = v.y;
      }
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) fma2(acc[i][j], a[i], b[j]);
    }
  }
  float out[TM][TN];
#pragma unroll
  for (int j = 0; j < TN; ++j)
#pragma unroll
    for (int i = 0; i < TM; ++i) out[i][j] = halves_sum(acc[i][j]);
  if constexpr (KG > 1) {
    // the groups' sums go through the first operand's stages, a few values of every lane at a time
    constexpr int LDR = TM * TN;                            // one lane's values
    float* sh = reinterpret_cast<float*>(&As[0]);
    __syncthreads();
    // value v of lane l of warp w (of the group): [group - 1][v][w][l], conflict-free
    constexpr int WL = WM * WN * 32;
    const int wl = (warp % (WM * WN)) * 32 + lane;
    constexpr int VP = (int)sizeof(As) / 4 / WL / (KG - 1);
    static_assert(VP >= 1, "at least one value per pass");
#pragma unroll
    for (int v0 = 0; v0 < LDR; v0 += VP) {
      if (kg > 0) {
#pragma unroll
        for (int v = v0; v < (v0 + VP < LDR ? v0 + VP : LDR); ++v)
          sh[((kg - 1) * VP + v - v0) * WL + wl] = out[v / TN][v % TN];
      }
      __syncthreads();
      if (kg == 0) {
#pragma unroll
        for (int v = v0; v < (v0 + VP < LDR ? v0 + VP : LDR); ++v)
#pragma unroll
          for (int g = 0; g < KG - 1; ++g)
            out[v / TN][v % TN] += sh[(g * VP + v - v0) * WL + wl];
      }
      __syncthreads();
    }
    if (kg > 0) return;
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int m = m0 + wm * 32 + (i >> 1) * 8 + ty * 2 + (i & 1);
#pragma unroll
    for (int j = 0; j < TN; j += 2) {
      const int n = n0 + wn * WTN + (j >> 1) * 16 + tx * 2;
      if (m < M && n < N) ep(m, n, out[i][j], out[i][j + 1], split);
    }
  }
  if constexpr (EP::COLSUM) {
    // the threads that fetched the same rows at different k add up, in order, through the second operand's stages
    static_assert(KG == 1 && !LB::K_CONTIG, "weight gradients");
    typedef FfLoader<LB, BN, BK, NT> FB;
    if (blockIdx.x == 0) {
      float4* sh = reinterpret_cast<float4*>(&Bs[0]);
      static_assert(FB::ITEMS * 16 <= sizeof(Bs), "fits");
      __syncthreads();
#pragma unroll
      for (int it = 0; it < FB::PER; ++it)
        if (FB::FULL || (int)threadIdx.x + it * NT < FB::ITEMS) sh[threadIdx.x + it * NT] = colsum[it];
      __syncthreads();
      if (threadIdx.x < BN / 4) {
        float4 t = sh[threadIdx.x];
        for (int q = 1; q < BK / 2; ++q) {
          const float4 v = sh[q * (BN / 4) + threadIdx.x];
          t.x += v.x; t.y += v.y; t.z += v.z; t.w += v.w;
        }
        const int n = n0 + threadIdx.x * 4;
        if (n < N) { ep.colsum(n, t.x, t.y, split); ep.colsum(n + 2, t.z, t.w, split); }
      }
    }
  }
}

// number of k blocks of BK a split covers when `splits` are asked for
inline int ffma_k_per_split(int K, int splits, int bk) { const int kps = (K + splits - 1) / splits; return (kps + bk - 1) / bk * bk; }

template <int WM, int WN, int TN, int KG, class LA, class LB, class EP>
inline void gemm_ffma(LaunchCtx& lc, int kid, int M, int N, int K, int k_per_split, int classes, LA la, LB lb, EP ep) {
  constexpr int BM = 32 * WM, BN = 8 * TN * WN;
  const int splits = (K + k_per_split - 1) / k_per_split;
  KernelScope scope(lc, kid);
  launch_kernel_overlapped(lc, gemm_ffma_kernel<WM, WN, TN, KG, LA, LB, EP>, dim3((M + BM - 1) / BM, (N + BN - 1) / BN, splits * classes),
                           dim3(32 * WM * WN * KG), 0, M, N, K, k_per_split, splits, la, lb, ep);
}

// ---- operands ------------------------------------------------------------------------------------------------------
// (enter(c): class c of a launch that runs several contractions side by side)
// x[row][k], rows ld apart
template <class T> struct FfRows {
  static constexpr bool K_CONTIG = true;
  typedef const T* Row;
  const T* p; int ld;
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ Row row(int r) const { return r >= 0 ? p + (size_t)r * ld : nullptr; }
  __device__ __forceinline__ float4 load(Row b, int k) const { return b ? load4(b + k) : make_float4(0.f, 0.f, 0.f, 0.f); }
};
// x[k][row]
template <class T> struct FfCols {
  static constexpr bool K_CONTIG = false;
  typedef const T* Row;
  const T* p; int ld;
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ Row row(int r) const { return r >= 0 ? p + r : nullptr; }
  __device__ __forceinline__ float4 load(Row b, int k) const { return b ? load4(b + (size_t)k * ld) : make_float4(0.f, 0.f, 0.f, 0.f); }
};
// convolution window: row = (state, oh, ow), k = (r, s, ci); the K C values of a filter row are contiguous
template <class G, class T> struct FfWindow {
  static constexpr bool K_CONTIG = true;
  typedef const T* Row;
  const T* x;
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ Row row(int m) const {
    if (m < 0) return nullptr;
    const int b = m / (G::OH * G::OW), rem = m % (G::OH * G::OW), oh = rem / G::OW, ow = rem % G::OW;
    return x + ((size_t)(b * G::H + oh * G::S) * G::W + ow * G::S) * G::C;
  }
  __device__ __forceinline__ float4 load(Row b, int k) const {
    return b ? load4(b + (k / (G::K * G::C)) * (G::W * G::C) + k % (G::K * G::C)) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
};
// the same window from the weight gradient: row j = (r, s, ci), k = (state, oh, ow)
template <class G, class T> struct FfWindowT {
  static constexpr bool K_CONTIG = false;
  typedef const T* Row;
  const T* x;
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ Row row(int j) const { return j >= 0 ? x + (j / (G::K * G::C)) * (G::W * G::C) + j % (G::K * G::C) : nullptr; }
  __device__ __forceinline__ float4 load(Row base, int m) const {
    if (!base) return make_float4(0.f, 0.f, 0.f, 0.f);
    const int b = m / (G::OH * G::OW), rem = m % (G::OH * G::OW), oh = rem / G::OW, ow = rem % G::OW;
    return load4(base + ((size_t)(b * G::H + oh * G::S) * G::W + ow * G::S) * G::C);
  }
};
// data gradient of a stride-1 layer: row = (state, y, x) of the layer input, k = (r, s, co); zero outside the output map
template <class G, class T> struct FfDgradWindow {
  static constexpr bool K_CONTIG = true;
  struct Row { const T* b; int y, x; };
  const T* g;
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ Row row(int m) const {
    if (m < 0) return Row{nullptr, 0, 0};
    const int b = m / (G::H * G::W), rem = m % (G::H * G::W);
    return Row{g + (size_t)b * G::OH * G::OW * G::CO, rem / G::W, rem % G::W};
  }
  __device__ __forceinline__ float4 load(const Row& q, int k) const {
    const int tap = k / G::CO, oh = q.y - tap / G::K, ow = q.x - tap % G::K;
    if (!q.b || (unsigned)oh >= (unsigned)G::OH || (unsigned)ow >= (unsigned)G::OW) return make_float4(0.f, 0.f, 0.f, 0.f);
    return load4(q.b + (oh * G::OW + ow) * G::CO + k % G::CO);
  }
};
template <class G, class T> struct FfWeightT {              // row = ci, k = (r, s, co)
  static constexpr bool K_CONTIG = false;
  typedef const T* Row;
  const T* w;
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ Row row(int r) const { return r >= 0 ? w + r : nullptr; }
  __device__ __forceinline__ float4 load(Row b, int k) const {
    return b ? load4(b + ((k % G::CO) * (G::K * G::K) + k / G::CO) * G::C) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
};
// Stride 2, 4 x 4 kernel: the input pixels of parity class (py, px) are touched by the four taps (py + 2 i, px + 2 j)
// only, a dense contraction of its own with a quarter of the reduction.  Row = (state, y >> 1, x >> 1), k = (i, j, co).
template <class G, class T> struct FfDgradClass {
  static constexpr bool K_CONTIG = true;
  struct Row { const T* b; int y, x; };
  const T* g;
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ Row row(int m) const {
    constexpr int HH = G::H / 2, WW = G::W / 2;
    if (m < 0) return Row{nullptr, 0, 0};
    const int b = m / (HH * WW), rem = m % (HH * WW);
    return Row{g + (size_t)b * G::OH * G::OW * G::CO, rem / WW, rem % WW};
  }
  __device__ __forceinline__ float4 load(const Row& q, int k) const {
    const int tap = k / G::CO, oh = q.y - (tap >> 1), ow = q.x - (tap & 1);
    if (!q.b || (unsigned)oh >= (unsigned)G::OH || (unsigned)ow >= (unsigned)G::OW) return make_float4(0.f, 0.f, 0.f, 0.f);
    return load4(q.b + (oh * G::OW + ow) * G::CO + k % G::CO);
  }
};
template <class G, class T> struct FfWeightClass {          // row = ci, k = (i, j, co) -> tap (py + 2 i, px + 2 j)
  static constexpr bool K_CONTIG = false;
  typedef const T* Row;
  const T* w; int z;
  __device__ __forceinline__ void enter(int c) { z = c; }
  __device__ __forceinline__ Row row(int r) const { return r >= 0 ? w + r + ((z >> 1) * G::K + (z & 1)) * G::C : nullptr; }
  __device__ __forceinline__ float4 load(Row b, int k) const {
    const int tap = k / G::CO;
    return b ? load4(b + (((k % G::CO) * G::K + 2 * (tap >> 1)) * G::K + 2 * (tap & 1)) * G::C) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
};

// ---- results -------------------------------------------------------------------------------------------------------
template <class T> struct FfBiasRelu {                       // out[m][n] = relu(acc * scale + bias[n])
  static constexpr bool COLSUM = false;
  T* out; const float* bias; int ld; float scale;
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ void operator()(int m, int n, float a, float b, int) const {
    store2(out + (size_t)m * ld + n, fmaxf(fmaf(a, scale, bias[n]), 0.f), fmaxf(fmaf(b, scale, bias[n + 1]), 0.f));
  }
};
template <class T> struct FfReluMask {                       // out[m][n] = act[m][n] > 0 ? acc : 0
  static constexpr bool COLSUM = false;
  T* out; const T* act; int ld;
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ void operator()(int m, int n, float a, float b, int) const {
    const size_t i = (size_t)m * ld + n;
    store2(out + i, to_f(act[i]) > 0.f ? a : 0.f, to_f(act[i + 1]) > 0.f ? b : 0.f);
  }
};
template <class G, class T> struct FfReluMaskClass {         // the same for parity class z: row (state, y >> 1, x >> 1)
  static constexpr bool COLSUM = false;
  T* out; const T* act; int z;
  __device__ __forceinline__ void enter(int c) { z = c; }
  __device__ __forceinline__ void operator()(int m, int n, float a, float b, int) const {
    constexpr int HH = G::H / 2, WW = G::W / 2;
    const int s = m / (HH * WW), rem = m % (HH * WW), y = 2 * (rem / WW) + (z >> 1), x = 2 * (rem % WW) + (z & 1);
    const size_t i = ((size_t)(s * G::H + y) * G::W + x) * G::C + n;
    store2(out + i, to_f(act[i]) > 0.f ? a : 0.f, to_f(act[i + 1]) > 0.f ? b : 0.f);
  }
};
struct FfPartial {                                           // part[split][m][n]
  static constexpr bool COLSUM = false;
  float* part; int M, N;
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ void operator()(int m, int n, float a, float b, int split) const {
    store2(part + ((size_t)split * M + m) * N + n, a, b);
  }
};
struct FfPartialColsum : FfPartial {                         // and the sum over k of B's rows: colpart[split][n]
  static constexpr bool COLSUM = true;
  float* colpart;
  __device__ __forceinline__ void colsum(int n, float a, float b, int split) const { store2(colpart + (size_t)split * N + n, a, b); }
};

}  // namespace paac

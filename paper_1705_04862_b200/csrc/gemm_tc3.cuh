// The float path's contractions on the tensor cores, accurate to float level:
//   C(m, n) = sum_k A(m, k) * B(n, k)
// with every float operand split into two TF32 pieces, x = hi + lo (hi = tf32(x), lo = tf32(x - hi), round to nearest,
// together 22 significant bits), and three tcgen05 passes (kind::tf32) per block of 32 k into a float accumulator in
// tensor memory, the blocks' sums then added in registers:
//   lo*hi + hi*lo + hi*hi      (the dropped lo*lo term and the rounding of lo are below 2^-21 of a product).
// Frame bytes and bf16 values are TF32 values as they are: they have no lo piece and need one pass less.
// Only the steps of one block are summed inside the tensor core, whose accumulation does not round to nearest;
// summed there over a whole contraction (thousands of steps) the result was eight times further from the exact
// one than the CUDA cores' chain of fused multiply-adds.
//
// Operands and epilogues are the functors of gemm_ffma.cuh.  A 128 x BN output tile per block and k split; 288 threads:
//   warps 0-7  fetch both operands' blocks as they are, by asynchronous copies T3_RING - 1 blocks ahead (neighbouring lanes take neighbouring
//              bytes: a lane per row of A cost 32 tag look-ups per load and set the kernel's pace, 93 us instead of
//              60 for the first layer's weight gradient over 640 states of the larger network).  Then a thread takes sixteen k of its row of A, splits them and stores the
//              pieces in tensor memory, where an operand of 128 rows lies as it is (row = lane, k = column): through shared memory, A's two
//              images would be written once and read three times, more bytes than the multiplications take time.  B's images go to shared
//              memory (128-byte rows, 128-byte swizzle).  Then the thread adds its columns of the finished product of the block
//              before to a running sum in registers.  At the end the sums pass through shared memory, so that results leave row by row.
//   warp 8     lane 0 issues the MMAs of a block (small terms first) into one of two accumulators, starting from zero, and commits.
// A stage's barrier `full` also says that the accumulator of the block before last has been read out (a warp arrives after it did),
// and `done` that the stage may be filled again, so two barriers per stage are all.  Two blocks are resident per SM: one splits
// while the other's multiplications run.  Every wait is bounded.
#pragma once
#include <cfloat>
#include <type_traits>

#include "gemm_ffma.cuh"
#include "tc_common.cuh"

namespace paac {

constexpr int T3_BM = 128, T3_BK = 32, T3_PWARPS = 8, T3_NT = T3_PWARPS * 32, T3_THREADS = T3_NT + 32, T3_KPT = 16, T3_RING = 3;
template <int BN> struct T3Cfg {
  static_assert(BN == 16 || BN == 32 || BN == 64, "tile width");
  static constexpr uint32_t IMAGE = BN * 128, STAGE = 2 * IMAGE, ACC0 = 2 * 2 * T3_BK, TMEM = 256;
  static constexpr int COLS = BN / 2, SLOTS = BN * 8, SLOTS_PER = (SLOTS + T3_NT - 1) / T3_NT, OUT_LD = BN + 4;
  static_assert(ACC0 + 2 * BN <= TMEM, "tensor memory: two stages of A's pieces and two accumulators, two blocks to an SM");
};
struct T3Shared {
  uint64_t full[2], done[2];
  uint32_t tmem_base;
  volatile uint32_t abort;
  uint32_t table[2][8][T3_BK];
};

// Instruction descriptor for kind::tf32: float accumulator, A and B in TF32 format (code 2), both K-major.
__host__ __device__ constexpr uint32_t make_idesc_tf32(int M, int N) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// D[tmem] (+)= A[tmem] * B[smem]: A's 128 rows in the lanes of a_tmem, eight k in as many columns; B's descriptor in two words
template <bool ACC>
__device__ __forceinline__ void mma_tf32_ts(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t b_hi, uint32_t idesc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\t"
      "setp.ne.b32 p, %5, 0;\n\t"
      "mov.b64 db, {%2, %3};\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], db, %4, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(b_hi), "r"(idesc), "n"(ACC ? 1 : 0)
      : "memory");
}
// sixteen columns of this warp's 32 lanes
__device__ __forceinline__ void t3_tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
        "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void t3_tmem_ld(uint32_t taddr, uint32_t (&r)[32]) { tc::tmem_ld_32x32(taddr, r); }
__device__ __forceinline__ void t3_tmem_ld(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]) : "r"(taddr) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void t3_tmem_ld(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// Two values x = hi + lo in TF32 pieces.  hi is rounded to nearest by integer arithmetic (the conversion takes three instructions for one).
// lo has up to twelve bits, of which the tensor cores read eleven: the factor brings what would be cut off up to a whole last place, so that lo
// is rounded too.  A NaN may be lost in hi, not in lo; an infinity gives a NaN (see the
// end of the kernel).
__device__ __forceinline__ void split_tf32(float x, float y, uint32_t& xh, uint32_t& yh, uint32_t& xl, uint32_t& yl) {
  xh = (__float_as_uint(x) + 0x1000u) & 0xFFFFE000u;
  yh = (__float_as_uint(y) + 0x1000u) & 0xFFFFE000u;
  asm("{\n\t.reg .b64 s, t, m, f;\n\tmov.b64 s, {%2, %3};\n\tmov.b64 t, {%4, %5};\n\tmov.b64 m, {%6, %6};\n\tmov.b64 f, {%7, %7};\n\t"
      "fma.rn.f32x2 s, t, m, s;\n\tmul.rn.f32x2 s, s, f;\n\tmov.b64 {%0, %1}, s;\n\t}"
      : "=r"(xl), "=r"(yl) : "f"(x), "f"(y), "r"(xh), "r"(yh), "f"(-1.f), "f"(1.f + 1.f / 2048.f));
}
__device__ __forceinline__ void t3_add2(float& x, float& y, uint32_t a, uint32_t b) {       // two additions in one instruction
  asm("{\n\t.reg .b64 s, t;\n\tmov.b64 s, {%0, %1};\n\tmov.b64 t, {%2, %3};\n\tadd.rn.f32x2 s, s, t;\n\tmov.b64 {%0, %1}, s;\n\t}"
      : "+f"(x), "+f"(y) : "r"(a), "r"(b));
}
template <class T> struct T3Exact { static constexpr bool value = true; };        // a TF32 value as it is
template <> struct T3Exact<float> { static constexpr bool value = false; };

// Where a thread's sixteen bytes of an operand lie in the block of 32 k from k0 on: a place of its own, worked out once (an element offset; no
// operand has 2^32), and what k0 adds for all.  Blocks never span two rows of a filter or two taps, and all operands but those of
// the weight gradients have a multiple of 32 k.  `taps`: bit t says whether tap t lies inside the map (data gradients).
struct T3Block { int off; uint32_t tap, inside; };  // what k0 adds; the tap; where tap 0 lies from there
template <class OP> struct T3Place {
  uint32_t off;
  __device__ __forceinline__ void init(const OP& op, int r, int k) { off = (uint32_t)(op.row(r) - op.any()) + (uint32_t)k; }
  static constexpr bool WHOLE = true;               // every piece lies inside
  __device__ __forceinline__ uint32_t at(const T3Block&, bool& in) const { in = true; return off; }
};
template <class G, int TAPS, int SIDE, class Row> __device__ __forceinline__ uint32_t t3_taps(const Row& q) {
  uint32_t taps = 0u;
#pragma unroll
  for (int t = 0; t < TAPS; ++t)
    if ((unsigned)(q.y - t / SIDE) < (unsigned)G::OH && (unsigned)(q.x - t % SIDE) < (unsigned)G::OW) taps |= 1u << t;
  return taps;
}
template <class OP, class G, int TAPS, int SIDE> struct T3DgradPlace {
  static constexpr bool WHOLE = false;
  uint32_t off, taps;
  __device__ __forceinline__ void init(const OP& op, int r, int k) {
    const auto q = op.row(r);
    off = (uint32_t)(q.b - op.any()) + (uint32_t)((q.y * G::OW + q.x) * G::CO + k);
    taps = t3_taps<G, TAPS, SIDE>(q);
  }
  __device__ __forceinline__ uint32_t at(const T3Block& b, bool& in) const {
    in = (taps >> b.tap) & 1u;
    return in ? off : b.inside;
  }
};
template <class G, class T> struct T3Place<FfDgradWindow<G, T>> : T3DgradPlace<FfDgradWindow<G, T>, G, G::K * G::K, G::K> {};
template <class G, class T> struct T3Place<FfDgradClass<G, T>> : T3DgradPlace<FfDgradClass<G, T>, G, 4, 2> {};
template <class G, int SIDE> __device__ __forceinline__ T3Block t3_dgrad_block(uint32_t k0) {
  static_assert(G::CO % T3_BK == 0, "blocks inside taps");
  const uint32_t tap = k0 / G::CO, shift = (tap / SIDE * G::OW + tap % SIDE) * G::CO;
  return {(int)(k0 % G::CO) - (int)shift, tap, shift};
}
template <class T> __device__ __forceinline__ T3Block t3_block(const FfRows<T>&, uint32_t k0) { return {(int)k0, 0u, 0u}; }
template <class G, class T> __device__ __forceinline__ T3Block t3_block(const FfWindow<G, T>&, uint32_t k0) {
  static_assert(G::K * G::C % T3_BK == 0, "blocks inside rows of the filter");
  return {(int)(k0 / (G::K * G::C) * (G::W * G::C) + k0 % (G::K * G::C)), 0u, 0u};
}
template <class G, class T> __device__ __forceinline__ T3Block t3_block(const FfDgradWindow<G, T>&, uint32_t k0) { return t3_dgrad_block<G, G::K>(k0); }
template <class G, class T> __device__ __forceinline__ T3Block t3_block(const FfDgradClass<G, T>&, uint32_t k0) { return t3_dgrad_block<G, 2>(k0); }
__device__ __forceinline__ void t3_copy16(uint32_t to, const void* from) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to), "l"(from) : "memory");
}
template <class T> __device__ __forceinline__ T t3_lds(uint32_t at);
template <> __device__ __forceinline__ uint4 t3_lds<uint4>(uint32_t at) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(at));
  return v;
}
template <> __device__ __forceinline__ uint2 t3_lds<uint2>(uint32_t at) {
  uint2 v;
  asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(at));
  return v;
}
template <> __device__ __forceinline__ uint32_t t3_lds<uint32_t>(uint32_t at) {
  uint32_t v;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(at));
  return v;
}
template <> __device__ __forceinline__ float t3_lds<float>(uint32_t at) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(at));
  return v;
}
template <> __device__ __forceinline__ bf16 t3_lds<bf16>(uint32_t at) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(at));
  return __ushort_as_bfloat16(v);
}
template <> __device__ __forceinline__ uint8_t t3_lds<uint8_t>(uint32_t at) {
  uint32_t v;
  asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(at));
  return (uint8_t)v;
}
template <class OP> __device__ __forceinline__ int t3_k_step(const OP& op) { return (int)(op.at(op.any(), 1) - op.at(op.any(), 0)); }      // inside a block

// The four parity classes of a stride-2 data gradient (FfDgradClass) read the same rows, so here they lie side by side along N: row = (class, ci)
// of the weights, column = (class, ci) of the result.
template <class G, class T> struct T3WeightClasses {
  static constexpr bool K_CONTIG = false;
  typedef T Elem;
  typedef const T* Row;
  const T* w;
  __device__ __forceinline__ const T* any() const { return w; }
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ Row row(int r) const { return w + (r / (2 * G::C) * G::K + r / G::C % 2) * G::C + r % G::C; }
  __device__ __forceinline__ const T* at(Row b, int k) const { return FfWeightClass<G, T>{w, 0}.at(b, k); }
};
template <class G, class T> struct T3ReluMaskClasses {
  static constexpr bool COLSUM = false;
  T* out; const T* act;
  __device__ __forceinline__ void enter(int) {}
  __device__ __forceinline__ void operator()(int m, int n, float4 v, int split) const { FfReluMaskClass<G, T>{out, act, n / G::C}(m, n % G::C, v, split); }
};
// Windows seen from the weight gradient: where a position's window starts takes divisions, so one warp works that out for a block.
template <class OP> struct T3Table { static constexpr bool use = false; };
template <class G, class T> struct T3Table<FfWindowT<G, T>> {
  static constexpr bool use = true;
  __device__ __forceinline__ static uint32_t offset(int m) {                      // (fewer than 2^32 elements)
    const int b = m / (G::OH * G::OW), rem = m % (G::OH * G::OW);
    return (uint32_t)((b * G::H + rem / G::OW * G::S) * G::W + rem % G::OW * G::S) * (uint32_t)G::C;
  }
};

// A block of 32 k of R rows as it lies in memory.  k contiguous: rows of 32 k, their 16-byte pieces permuted so that eight neighbouring rows'
// pieces of the same k lie in different banks; else [k][R].  Rows past the last one repeat it (or its piece): their results are dropped.
template <class OP, int R, bool K_CONTIG = OP::K_CONTIG> struct T3Raw {
  typedef typename OP::Elem T;
  static constexpr int V = 16 / (int)sizeof(T), ITEMS = R * T3_BK / V, PER = (ITEMS + T3_NT - 1) / T3_NT, BYTES = R * T3_BK * (int)sizeof(T);
  static constexpr int PIECES = T3_BK / V;                                        // of a row
  T3Place<OP> place[PER];
  uint32_t to0;                                                                   // where this thread's first piece goes
  __device__ __forceinline__ static uint32_t piece_at(int r, int c) {
    return (uint32_t)(r * PIECES + (c ^ ((r / (8 / PIECES)) & (PIECES - 1)))) * 16u;
  }
  __device__ __forceinline__ void init(const OP& op, int r0, int rows) {
    to0 = piece_at((int)threadIdx.x / PIECES, (int)threadIdx.x % PIECES);
#pragma unroll
    for (int it = 0; it < PER; ++it) {
      const int i = (int)threadIdx.x + it * T3_NT;
      place[it].init(op, min(r0 + i / PIECES, rows - 1), i % PIECES * V);
    }
  }
  __device__ __forceinline__ void fetch(const OP& op, int k0, int, uint32_t to, const uint32_t*) const {
    const T3Block b = t3_block(op, (uint32_t)k0);
    const T* base = op.any() + b.off;
    static_assert(T3_NT / PIECES % 8 == 0, "a thread's pieces have one permutation");
#pragma unroll
    for (int it = 0; it < PER; ++it) {
      if (ITEMS % T3_NT != 0 && (int)threadIdx.x + it * T3_NT >= ITEMS) break;
      bool in;
      const uint32_t off = place[it].at(b, in);
      if constexpr (T3Place<OP>::WHOLE) t3_copy16(to + to0 + it * (T3_NT * 16), base + off);
      else tc::cp_async16(to + to0 + it * (T3_NT * 16), base + off, in ? 16u : 0u);
    }
  }
  // N neighbouring k, from k on, of one row: where that is, and the values of a block at `raw`
  struct Reader {
    uint32_t at;                                       // of the first piece; the others' lie a bit pattern away
    __device__ __forceinline__ void init(int r, int k) { at = piece_at(r, k / V) + k % V * (int)sizeof(T); }
  };
  template <int N> __device__ __forceinline__ static void read(const Reader& rd, uint32_t raw, float (&x)[N]) {
    if constexpr (N < V) {
      static_assert(N == 4 && sizeof(T) <= 2, "part of a piece");
      float4 f;
      if constexpr (sizeof(T) == 2) f = widen4(t3_lds<uint2>(raw + rd.at));
      else f = widen4(t3_lds<uint32_t>(raw + rd.at));
      x[0] = f.x; x[1] = f.y; x[2] = f.z; x[3] = f.w;
    } else {
#pragma unroll
      for (int c = 0; c < N / V; ++c) {
        float4 f[V / 4];
        widen(t3_lds<uint4>(raw + (rd.at ^ (uint32_t)(c * 16))), (const T*)nullptr, f);
#pragma unroll
        for (int q = 0; q < V / 4; ++q) {
          float* to = x + c * V + 4 * q;
          to[0] = f[q].x; to[1] = f[q].y; to[2] = f[q].z; to[3] = f[q].w;
        }
      }
    }
  }
};
template <class OP, int R> struct T3Raw<OP, R, false> {
  typedef typename OP::Elem T;
  static constexpr int V = 16 / (int)sizeof(T), ITEMS = R * T3_BK / V, PER = (ITEMS + T3_NT - 1) / T3_NT, BYTES = R * T3_BK * (int)sizeof(T);
  static constexpr int GROUPS = R / V;                                            // of rows
  static_assert(T3_NT % GROUPS == 0, "a thread keeps its rows");
  static constexpr int K_OF = T3_NT / GROUPS;                                     // k from one of a thread's pieces to the next
  uint32_t off, step, k;
  __device__ __forceinline__ void init(const OP& op, int r0, int rows) {
    k = threadIdx.x / GROUPS;
    off = (uint32_t)(op.row(min(r0 + (int)threadIdx.x % GROUPS * V, rows - V)) - op.any());
    if constexpr (!T3Table<OP>::use) { step = (uint32_t)t3_k_step(op); off += k * step; }
  }
  __device__ __forceinline__ void fetch(const OP& op, int k0, int k_end, uint32_t to, const uint32_t* table) const {
    const T* base = op.any();
    if constexpr (!T3Table<OP>::use) base = op.at(base, k0);
    const uint32_t left = (uint32_t)(k_end - k0);
#pragma unroll
    for (int it = 0; it < PER; ++it) {
      const int i = (int)threadIdx.x + it * T3_NT;
      if (ITEMS % T3_NT != 0 && i >= ITEMS) break;
      const bool in = k + it * K_OF < left;
      const uint32_t from = T3Table<OP>::use ? off + table[k + it * K_OF] : off + it * K_OF * step;
      tc::cp_async16(to + (uint32_t)i * 16u, base + (in ? from : 0u), in ? 16u : 0u);
    }
  }
  struct Reader {
    uint32_t at;
    __device__ __forceinline__ void init(int r, int k) { at = (uint32_t)(k * R + r) * (uint32_t)sizeof(T); }
  };
  template <int N> __device__ __forceinline__ static void read(const Reader& rd, uint32_t raw, float (&x)[N]) {
#pragma unroll
    for (int j = 0; j < N; ++j) x[j] = to_f(t3_lds<T>(raw + rd.at + j * R * (int)sizeof(T)));
  }
};
__device__ __forceinline__ void t3_sync() { asm volatile("bar.sync 1, %0;" ::"n"(T3_NT) : "memory"); }      // the eight warps
__device__ __forceinline__ bool t3_any(bool mine) {               // the same, and whether any thread says so
  uint32_t any;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\tbar.red.or.pred p, 1, %2, q;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(any) : "r"(mine ? 1u : 0u), "n"(T3_NT) : "memory");
  return any != 0u;
}

template <int BN, class LA, class LB, class EP>
__global__ void __launch_bounds__(T3_THREADS, 2)
gemm_tc3_kernel(int M, int N, int K, int k_per_split, int splits, LA la, LB lb, EP ep, uint32_t* error_word) {
  using namespace tc;
  typedef T3Cfg<BN> C;
  constexpr bool A_EXACT = T3Exact<typename LA::Elem>::value, B_EXACT = T3Exact<typename LB::Elem>::value;
  typedef T3Raw<LA, T3_BM> RawA;
  typedef T3Raw<LB, BN> RawB;
  constexpr uint32_t RAW = RawA::BYTES + RawB::BYTES;
  extern __shared__ __align__(16) uint8_t dyn_smem[];
  __shared__ T3Shared sh;
  uint8_t* const images = dyn_smem + ((1024u - (smem_u32(dyn_smem) & 1023u)) & 1023u);
  uint8_t* const raws = images + 2 * C::STAGE;
  const uint32_t b_base = smem_u32(images), raw_base = smem_u32(raws);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.x * T3_BM, n0 = blockIdx.y * BN, split = blockIdx.z % splits, cls = blockIdx.z / splits;
  const int k_begin = split * k_per_split, k_end = min(K, k_begin + k_per_split);
  const int num_kb = k_end > k_begin ? (k_end - k_begin + T3_BK - 1) / T3_BK : 0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) { mbar_init(&sh.full[s], T3_PWARPS); mbar_init(&sh.done[s], 1); }
    sh.abort = 0u;
    fence_barrier_init();
  }
  if (warp == T3_PWARPS) tmem_alloc(&sh.tmem_base, C::TMEM);
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  const uint32_t tmem = sh.tmem_base;
  pdl_entry();          // everything above touches only this block's own resources
  la.enter(cls); lb.enter(cls); ep.enter(cls);

  if (warp < T3_PWARPS) {
    const int quarter = warp & 3, grp = warp >> 2;
    const uint32_t lanes = (uint32_t)(32 * quarter) << 16;
    RawA a;
    RawB b;
    a.init(la, m0, M);
    b.init(lb, n0, N);
    // B is split in slots of four k of one column: eight neighbouring threads share a column where k is contiguous, else 32 take 32 columns
    int b_col[C::SLOTS_PER], b_k[C::SLOTS_PER];
    uint32_t b_to[C::SLOTS_PER];
    typename RawB::Reader b_from[C::SLOTS_PER];
    typename RawA::Reader a_from;
    a_from.init(32 * quarter + lane, T3_KPT * grp);
    float colsum[C::SLOTS_PER];
#pragma unroll
    for (int i = 0; i < C::SLOTS_PER; ++i) {
      const int slot = (int)threadIdx.x + i * T3_NT;
      b_col[i] = LB::K_CONTIG ? slot >> 3 : slot & (BN - 1);
      b_k[i] = 4 * (LB::K_CONTIG ? slot & 7 : slot / BN);
      b_from[i].init(b_col[i], b_k[i]);
      b_to[i] = b_base + sw128_offset((uint32_t)b_col[i], (uint32_t)b_k[i] >> 2);
      colsum[i] = 0.f;
    }
    constexpr bool TABLE = T3Table<LA>::use;
    auto tabulate = [&](int group) {                   // of eight blocks, an entry to a thread
      if constexpr (TABLE)
        sh.table[group & 1][0][threadIdx.x] = T3Table<LA>::offset(k_begin + group * (8 * T3_BK) + (int)threadIdx.x);
    };
    auto fetch = [&](int kb, uint32_t to) {
      if (kb < num_kb) {
        a.fetch(la, k_begin + kb * T3_BK, k_end, to, sh.table[kb >> 3 & 1][kb & 7]);
        b.fetch(lb, k_begin + kb * T3_BK, k_end, to + RawA::BYTES, nullptr);
      }
      cp_async_commit();
    };
    float sum[C::COLS];
#pragma unroll
    for (int j = 0; j < C::COLS; ++j) sum[j] = 0.f;
    bool alive = true;
    // adds the finished product of block `kb` to the running sum
    auto collect = [&](int kb) {
      const bool ok = mbar_wait(&sh.done[kb & 1], (kb >> 1) & 1, &sh.abort, error_word, ERR_WAIT_ACC);
      if (!__all_sync(0xffffffffu, ok)) return false;
      tcgen05_fence_after();
      uint32_t r[C::COLS];
      t3_tmem_ld(tmem + lanes + C::ACC0 + (kb & 1) * BN + grp * C::COLS, r);
#pragma unroll
      for (int j = 0; j < C::COLS; j += 2) t3_add2(sum[j], sum[j + 1], r[j], r[j + 1]);
      return true;
    };
    static_assert(T3_RING == 3 && T3_NT == 8 * T3_BK, "two blocks are on their way; eight blocks to a table");
    if constexpr (TABLE) { tabulate(0); t3_sync(); }
    fetch(0, raw_base);
    fetch(1, raw_base + RAW);
    uint32_t at_raw = 0u, at_next = 2u * RAW;          // of the ring: block kb, and block kb + 2
    for (int kb = 0; kb < num_kb; ++kb) {
      const int s = kb & 1;
      cp_async_wait<T3_RING - 2>();
      t3_sync();                     // block kb is in; everyone is done with what block kb - 1 was split from
      fetch(kb + 2, raw_base + at_next);
      if (TABLE && (kb & 7) == 0) tabulate((kb >> 3) + 1);      // (read from six blocks on)
      const uint32_t raw = raw_base + at_raw;
      at_next = at_raw;
      at_raw = at_raw == 2u * RAW ? 0u : at_raw + RAW;
      {
        float x[T3_KPT];
        uint32_t hi[T3_KPT], lo[T3_KPT];
        RawA::read(a_from, raw, x);
        const uint32_t at = tmem + lanes + s * (2 * T3_BK) + T3_KPT * grp;
#pragma unroll
        for (int j = 0; j < T3_KPT; j += 2) {
          if constexpr (A_EXACT) { hi[j] = __float_as_uint(x[j]); hi[j + 1] = __float_as_uint(x[j + 1]); }
          else split_tf32(x[j], x[j + 1], hi[j], hi[j + 1], lo[j], lo[j + 1]);
        }
        t3_tmem_st16(at, hi);
        if constexpr (!A_EXACT) t3_tmem_st16(at + T3_BK, lo);
      }
#pragma unroll
      for (int i = 0; i < C::SLOTS_PER; ++i) {
        if (C::SLOTS % T3_NT != 0 && (int)threadIdx.x >= C::SLOTS) break;
        float x[4];
        uint32_t hi[4], lo[4];
        RawB::read(b_from[i], raw + RawA::BYTES, x);
        const uint32_t to = b_to[i] + s * C::STAGE;
#pragma unroll
        for (int j = 0; j < 4; j += 2) {
          if constexpr (B_EXACT) { hi[j] = __float_as_uint(x[j]); hi[j + 1] = __float_as_uint(x[j + 1]); }
          else split_tf32(x[j], x[j + 1], hi[j], hi[j + 1], lo[j], lo[j + 1]);
        }
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(to), "r"(hi[0]), "r"(hi[1]), "r"(hi[2]), "r"(hi[3]) : "memory");
        if constexpr (!B_EXACT)
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(to + C::IMAGE), "r"(lo[0]), "r"(lo[1]), "r"(lo[2]), "r"(lo[3]) : "memory");
        if constexpr (EP::COLSUM) colsum[i] += (x[0] + x[1]) + (x[2] + x[3]);
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      fence_proxy_async_smem();
      tcgen05_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.full[s]);
      if (alive && kb >= 1) alive = collect(kb - 1);              // (a warp that gave up goes on without waiting: the others meet it above)
    }
    if (alive && num_kb > 0) alive = collect(num_kb - 1);
    cp_async_wait<0>();
    bool finite = true;
#pragma unroll
    for (int j = 0; j < C::COLS; ++j) finite = finite && fabsf(sum[j]) <= FLT_MAX;
    if (t3_any(alive && !finite)) {  // (the ring is free, and the instructions are through with the images)
      // An infinity, or a value that rounds to one, has no lo piece: where a sum is not finite, the tile is done again by chains of fused
      // multiply-adds, as the CUDA cores would have done it.
#pragma unroll
      for (int j = 0; j < C::COLS; ++j) sum[j] = 0.f;
      for (int kb = 0; kb < num_kb; ++kb) {
        if (TABLE && (kb & 7) == 0) tabulate(kb >> 3);
        t3_sync();                   // the table is in, and everyone is done with the block before
        fetch(kb, raw_base);
        cp_async_wait<0>();
        t3_sync();
#pragma unroll 1
        for (int k = 0; k < T3_BK; k += 4) {
          typename RawA::Reader from_a;
          float x[4];
          from_a.init(32 * quarter + lane, k);
          RawA::read(from_a, raw_base, x);
#pragma unroll
          for (int j = 0; j < C::COLS; ++j) {
            typename RawB::Reader from_b;
            float y[4];
            from_b.init(grp * C::COLS + j, k);
            RawB::read(from_b, raw_base + RawA::BYTES, y);
#pragma unroll
            for (int q = 0; q < 4; ++q) sum[j] = fmaf(x[q], y[q], sum[j]);
          }
        }
      }
      t3_sync();
    }
    float* out = reinterpret_cast<float*>(raws);
#pragma unroll
    for (int j = 0; j < C::COLS; j += 4)
      *reinterpret_cast<float4*>(out + (32 * quarter + lane) * C::OUT_LD + grp * C::COLS + j) = make_float4(sum[j], sum[j + 1], sum[j + 2], sum[j + 3]);
    float* cs = out + T3_BM * C::OUT_LD;
    if constexpr (EP::COLSUM) {
      static_assert(!LB::K_CONTIG, "weight gradients");
#pragma unroll
      for (int i = 0; i < C::SLOTS_PER; ++i)
        if ((int)threadIdx.x + i * T3_NT < C::SLOTS) cs[(b_k[i] >> 2) * BN + b_col[i]] = colsum[i];
    }
    t3_sync();
    if (sh.abort == 0u) {
#pragma unroll 2
      for (int i = threadIdx.x; i < T3_BM * BN / 4; i += T3_NT) {
        const int r = i / (BN / 4), n = n0 + i % (BN / 4) * 4;
        if (m0 + r < M && n < N) ep(m0 + r, n, *reinterpret_cast<const float4*>(out + r * C::OUT_LD + n - n0), split);
      }
      if constexpr (EP::COLSUM) {
        if (blockIdx.x == 0 && threadIdx.x < BN && n0 + (int)threadIdx.x < N) {
          float t = 0.f;                                           // the eight groups of four k, in order
#pragma unroll
          for (int q = 0; q < 8; ++q) t += cs[q * BN + threadIdx.x];
          ep.colsum(n0 + threadIdx.x, t, split);
        }
      }
    }
  } else if (lane == 0) {
    // ---------------- MMA issuer ----------------
    constexpr uint32_t idesc = make_idesc_tf32(T3_BM, BN);
    const uint32_t desc_word = desc_hi_kmajor_sw128();
    for (int kb = 0; kb < num_kb; ++kb) {
      const int s = kb & 1;
      if (!mbar_wait(&sh.full[s], (kb >> 1) & 1, &sh.abort, error_word, ERR_WAIT_FULL)) break;
      tcgen05_fence_after();
      const uint32_t d = tmem + C::ACC0 + s * BN, a_hi = tmem + s * (2 * T3_BK), a_lo = a_hi + T3_BK;
      const uint32_t b_hi = ((b_base + s * C::STAGE) >> 4) & 0x3FFFu, b_lo = b_hi + (C::IMAGE >> 4);
      auto pass = [&](auto first, uint32_t pa, uint32_t pb) {
        mma_tf32_ts<!decltype(first)::value>(d, pa, pb, desc_word, idesc);
#pragma unroll
        for (int k = 1; k < T3_BK / 8; ++k) mma_tf32_ts<true>(d, pa + 8 * k, pb + 2 * k, desc_word, idesc);
      };
      if constexpr (!A_EXACT) pass(std::true_type{}, a_lo, b_hi);                    // small terms first
      if constexpr (!B_EXACT) pass(std::integral_constant<bool, A_EXACT>{}, a_hi, b_lo);
      pass(std::integral_constant<bool, A_EXACT && B_EXACT>{}, a_hi, b_hi);
      mma_commit(&sh.done[s]);
    }
  }
  tcgen05_fence_before();
  __syncthreads();
  if (warp == T3_PWARPS) {
    __syncwarp();
    tcgen05_fence_after();
    tmem_dealloc(tmem, C::TMEM);
  }
}

template <int BN, class LA, class LB, class EP>
inline void gemm_tc3(LaunchCtx& lc, int kid, int M, int N, int K, int k_per_split, int classes, LA la, LB lb, EP ep) {
  // the images, then the larger of the ring and the sums' tile
  constexpr int ring = T3_RING * (T3Raw<LA, T3_BM>::BYTES + T3Raw<LB, BN>::BYTES), sums = T3_BM * T3Cfg<BN>::OUT_LD * 4 + 8 * BN * 4;
  constexpr int smem = 1024 + 2 * (int)T3Cfg<BN>::STAGE + (ring > sums ? ring : sums);
  static_assert(2 * smem <= 226 * 1024, "two blocks to an SM");
  auto kern = gemm_tc3_kernel<BN, LA, LB, EP>;
  static const cudaError_t attr = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (attr != cudaSuccess) lc.host_failure = true;
  const int splits = (K + k_per_split - 1) / k_per_split;
  KernelScope scope(lc, kid);
  launch_kernel_overlapped(lc, kern, dim3((M + T3_BM - 1) / T3_BM, (N + BN - 1) / BN, splits * classes), dim3(T3_THREADS), smem, M, N, K,
                           k_per_split, splits, la, lb, ep, lc.error_word);
}

}  // namespace paac

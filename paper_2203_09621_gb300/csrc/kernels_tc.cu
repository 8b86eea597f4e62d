// Dual-precision layer product on the sm_103a tensor cores (tcgen05 + TMEM
// + TMA), with the SP2 layer update fused into the epilogue.
//
// What one launch computes (one deep layer of Sec. III, Algorithm 1):
//   square   (job 0):   X  = S0 S0             ~ hi*hi + hi*lo + lo*hi
//                       (Sec. II C, Eq. (S0 tensor core): A + B + B^T)
//   response (job 1+k): X1 = S0 S1_k + S1_k S0 ~ sum of the 3-term dual
//                       products of both orders (Sec. III D,
//                       Eq. (FP32S0S1), Eq. (S0S1 tensor core))
// each accumulated in FP32 in tensor memory, and then
//   S_n = sigma X + (1 - sigma) S_{n-1}      (Eq. (eq:Sn); Alg. 2 and 3)
// written as an FP32 master plus its new hi/lo split (Eq. (DualMat2)).
//
// Symmetry (Sec. III D): every S is symmetric, so the B operand of a row
// block product can be read as a row panel (B[k][j] = B[j][k], "K-major"
// for both operands) and only tiles holding elements with row <= col are
// computed; the epilogue stores each such element at (r, c) and (c, r).
// The response needs both orders S0 S1 and S1 S0 for a tile, which are two
// K passes into the same accumulator.
//
// Kernel structure (persistent, one CTA per SM, 320 threads):
//   warp 0      TMA producer: 4-stage ring of {A_hi, A_lo, B_hi, B_lo}
//               tiles (128x32, 128x32, 256x32, 256x32 16-bit, 64B swizzle)
//   warp 1      TMEM owner and MMA issuer: tcgen05.mma.cta_group::1
//               kind::f16, M = 128, N = 256, K = 16, FP32 accumulate, two
//               256-column accumulators in TMEM (double buffered)
//   warps 2..9  epilogue: two warps per TMEM lane quadrant, one row and one
//               column half per thread; fused update, stores, deterministic
//               FP64 partial norms per tile
// Accumulation in chunks: the tensor core adds each MMA's products into the
// FP32 accumulator with a truncating alignment, so an error that grows with
// the number of MMAs folded into one accumulator (and is biased) would
// build up over K = 3n terms.  The K sequence of a tile is therefore cut into
// chunks of `chunk` stages (default 256 K-elements); each chunk starts a
// fresh TMEM accumulator and the epilogue warps add the chunk results in
// FP32 with round-to-nearest in registers.  The two TMEM accumulators are
// used alternately, so the MMA of the next chunk overlaps that summation.
// Every mbarrier wait is bounded in time; on expiry the CTA raises
// State::timeout_flag, drains its copies in flight (bounded), frees TMEM and
// returns, and the host reports DMPT_ETIMEOUT.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <math.h>

#include <mutex>
#include <type_traits>

#include "dmpt_internal.cuh"

namespace dmpt {
namespace tc {

constexpr int BM = 128;          // rows per tile (TMEM lanes)
constexpr int BN = 256;          // columns per tile
constexpr int BK = 32;           // K elements per stage (64 B rows)
constexpr int STAGES = 4;
constexpr int A_BYTES = BM * BK * 2;   // 8 KB
constexpr int B_BYTES = BN * BK * 2;   // 16 KB
constexpr int STAGE_BYTES = 2 * A_BYTES + 2 * B_BYTES;  // 48 KB
constexpr int TMEM_COLS = 512;   // two accumulators of BN columns
constexpr int EPI_WARPS = 8;     // two per TMEM lane quadrant (column halves)
constexpr int EPI_THREADS = 32 * EPI_WARPS;
constexpr int EPI_WARP0 = 2;     // epilogue = warps 2 .. 9
constexpr int NUM_THREADS = 64 + EPI_THREADS;
// Epilogue scratch: the partial sums of a tile (tile_sums_out), then one
// 32 x 32 block of 16-bit values per epilogue warp, its rows padded to DLD.
constexpr int EPI_SUMS = 512;
constexpr int DLD = 34;
constexpr int EPI_SCRATCH = EPI_SUMS + EPI_WARPS * 32 * DLD * 2;
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 /* align */ + 1024 /* barriers etc */ +
                           EPI_SCRATCH;
constexpr int DEFAULT_CHUNK_K = 256;  // K elements per tensor-memory accumulation chunk

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
      "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]),
      "f"(v[8]), "f"(v[9]), "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]),
      "f"(v[15])
      : "memory");
}

// ---------------------------------------------------------------------------
// PTX helpers

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint64_t gtimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait: false when `limit_ns` passes or another role of this CTA
// has aborted.  On expiry it raises both abort flags.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint64_t limit_ns,
                                          volatile int* abort_smem, int* timeout_global) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = gtimer();
  uint32_t it = 0;
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((++it & 255) == 0) {
      if (*abort_smem) return false;
      if (gtimer() - t0 > limit_ns) {
        *abort_smem = 1;
        atomicExch(timeout_global, 1);
        return false;
      }
    }
  }
}

// One lane of a converged warp, the same one each time.  Code under it stays
// warp-uniform for the compiler, so the operands of the tensor-core and TMA
// instructions need no per-lane handling (see mma_item).
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(p));
  return p != 0;
}

// mbar_wait by a whole converged warp: every lane gets the same answer.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, uint64_t limit_ns,
                                               volatile int* abort_smem, int* timeout_global) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  const uint64_t t0 = gtimer();
  uint32_t it = 0;
  while (true) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    if ((++it & 255) == 0) {
      const bool late = gtimer() - t0 > limit_ns;
      if (__any_sync(0xffffffffu, late || *abort_smem)) {
        if (late) {
          *abort_smem = 1;
          atomicExch(timeout_global, 1);
        }
        return false;
      }
    }
  }
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y,
                                            int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

__device__ __forceinline__ void fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Shared-memory matrix descriptor, K-major operand with 64-byte swizzle:
// rows of 64 B, 8-row groups 512 B apart (SBO), version 1, layout 4.
__device__ __forceinline__ uint64_t sw64_desc(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;             // LBO (unused for swizzled K-major)
  d |= (uint64_t)(512 >> 4) << 32;    // SBO
  d |= (uint64_t)1 << 46;             // descriptor version
  d |= (uint64_t)4 << 61;             // SWIZZLE_64B
  return d;
}

// The same with 128-byte swizzle: rows of 128 B, 8-row groups 1024 B apart,
// layout 2.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;             // LBO (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;   // SBO
  d |= (uint64_t)1 << 46;             // descriptor version
  d |= (uint64_t)2 << 61;             // SWIZZLE_128B
  return d;
}

// Instruction descriptor, kind::f16: D = F32, A/B = F16 (0) or BF16 (1),
// both K-major, N = 256, M = 128.
__host__ __device__ constexpr uint32_t make_idesc(int ab_type) {
  return (1u << 4) | ((uint32_t)ab_type << 7) | ((uint32_t)ab_type << 10) |
         ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}

__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
      : "memory");
}

// FP16 / BF16 rounding (round to nearest even) used by the dual split.
template <bool BF>
struct Cvt;
template <>
struct Cvt<false> {
  using T = __half;
  static __device__ __forceinline__ uint32_t pack(float a, float b) {   // a in the low half
    const __half2 v = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&v);
  }
  static __device__ __forceinline__ void unpack(uint32_t v, float& a, float& b) {
    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&v));
    a = f.x;
    b = f.y;
  }
};
template <>
struct Cvt<true> {
  using T = __nv_bfloat16;
  static __device__ __forceinline__ uint32_t pack(float a, float b) {   // a in the low half
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&v);
  }
  static __device__ __forceinline__ void unpack(uint32_t v, float& a, float& b) {
    a = __uint_as_float(v << 16);
    b = __uint_as_float(v & 0xffff0000u);
  }
};

// AND of a predicate over the epilogue threads (named barrier 1).
__device__ __forceinline__ int epi_all(int pred) {
  int out;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 q, %1, 0;\n\t"
      "bar.red.and.pred p, 1, %2, q;\n\t"
      "selp.s32 %0, 1, 0, p;\n\t}"
      : "=r"(out)
      : "r"(pred), "n"(EPI_THREADS)
      : "memory");
  return out;
}
__device__ __forceinline__ void epi_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(EPI_THREADS) : "memory");
}

// ---------------------------------------------------------------------------
// Work items: (job, tile).  Tiles: 128-row block I and 256-column block J
// with I <= 2J + 1 (the tile holds some element with row <= col).  Tile t
// is J-major: tiles of column block J are t = J(J+1) ... J(J+1) + 2J + 1.

__host__ __device__ inline int64_t num_tiles(int64_t Np) {
  const int64_t tj = Np / BN;
  return tj * (tj + 1);
}
__device__ __forceinline__ void tile_coords(int64_t t, int* I, int* J) {
  int j = (int)((sqrt(4.0 * (double)t + 1.0) - 1.0) * 0.5);
  while ((int64_t)(j + 1) * (j + 2) <= t) ++j;
  while ((int64_t)j * (j + 1) > t) --j;
  *J = j;
  *I = (int)(t - (int64_t)j * (j + 1));
}

// Jobs of a layer as a bit mask: bit 0 = square, bit 1 + j = response j.
// Item order: responses (ascending j) first, then the square.
__device__ __forceinline__ int job_at(uint32_t mask, int idx) {
  const uint32_t resp = mask & ~1u;
  const int nresp = __popc(resp);
  if (idx >= nresp) return 0;
  uint32_t m = resp;
  for (int i = 0; i < idx; ++i) m &= m - 1;  // drop the lowest set bits
  return __ffs(m) - 1;
}

// Jobs of a layer: 0 = square of S0; 1 + (o - 1) k1 + d = the order-o term
// of direction d (o = 1 .. order, d = 0 .. k1 - 1; k1 = first-order
// directions), whose activation is (Sec. III A, Eq. (S_n detailed))
//   S0 S_o + S_o S0 + sum_{a=1}^{o-1} S_a S_{o-a}
// in o + 1 K passes: pass 0 = S0 S_o, pass 1 = S_o S0, pass p >= 2 =
// S_{p-1} S_{o-p+1} (order 1: S0 S1, S1 S0; order 2 adds S1 S1).
// The job id is also the matrix slot of the result.
__device__ __forceinline__ int job_order(int job, int k1) { return 1 + (job - 1) / k1; }
__device__ __forceinline__ int job_passes(int job, int k1) {
  return job == 0 ? 1 : (job <= k1 ? 2 : 1 + job_order(job, k1));
}
// slot of the order-a term (a >= 1) of the direction of job `job`
__device__ __forceinline__ int job_slot(int job, int a, int k1) {
  return 1 + (a - 1) * k1 + (job - 1) % k1;
}
// operand slots (A, B) of pass `pass` of job `job`
__device__ __forceinline__ void job_operands(int job, int pass, int k1, int* mA, int* mB) {
  if (job == 0) {
    *mA = 0;
    *mB = 0;
  } else if (pass == 0) {
    *mA = 0;
    *mB = job;
  } else if (pass == 1) {
    *mA = job;
    *mB = 0;
  } else {
    *mA = job_slot(job, pass - 1, k1);
    *mB = job_slot(job, job_order(job, k1) - pass + 1, k1);
  }
}
// exact power-of-two unscale of a pass p >= 2 product (operands scaled by
// 2^e of their slots)
__device__ __forceinline__ float cross_unscale(const State* st, int job, int pass, int k1) {
  int mA, mB;
  job_operands(job, pass, k1, &mA, &mB);
  return ldexpf(1.0f, -(st->s1_exp_cur[mA - 1] + st->s1_exp_cur[mB - 1]));
}
// K range of the products: the 32-wide K blocks that hold columns < n.  The
// blocks of the padding to Np hold zeros on both sides and are left out
// (n = 5904: 185 of 192 blocks, solve 57.4 -> 54.4 ms).  The accumulation
// chunks keep the boundaries they have over all Np / 32 blocks, so results do
// not change: a backwards sweep starts `kchunk0` stages into its first chunk.
__host__ __device__ __forceinline__ int k_blocks(int64_t n) { return (int)((n + BK - 1) / BK); }

// Columns of a tile (width nt, from column c) left of cend = 32 k_blocks(n).
// Columns and rows from cend on are neither computed nor stored: as K range
// they are left out, and as rows of a tile they only reach elements that are
// left out as well, so they may hold anything.  The tiles of the last column
// block shrink their MMAs' N to what is left: n = 5904 (32 of 256 columns in 24
// of 300 tiles) 53.3 -> 52.5 ms, 32 uneven instances 18.3 -> 17.2 ms.
__host__ __device__ __forceinline__ int tile_cols(int c, int nt, int cend) {
  const int w = cend - c;
  return w < 0 ? 0 : (w < nt ? w : nt);
}
__device__ __forceinline__ int kchunk0(int64_t Np, int kblocks, int chunk, bool rev) {
  return rev ? ((int)(Np / BK) - kblocks) % chunk : 0;
}

// K-pass of accumulation chunk c (chunks never straddle passes); the
// producer of the pair kernel runs the passes backwards in odd rounds
__device__ __forceinline__ int chunk_pass(int c, int cpp, int passes, bool rev) {
  const int p = c / cpp;
  return rev ? passes - 1 - p : p;
}

// Operand slice of matrix m: S0 comes from the slice the control block
// names (ping-pong slot, or a tape slice when the S0 states are kept for the
// adjoint); S1_j from its ping-pong slot.
__device__ __forceinline__ int zop(int m, int buf, int part, int k, int z0) {
  return m == 0 ? z0 + part : zslice(buf, m, part, k);
}

// (s, c) += (s2, c2): sums held as s + c, the rounding of s kept in c (TwoSum)
__device__ __forceinline__ void ff_add(float& s, float& c, float s2, float c2) {
  const float t = s + s2;
  const float b = t - s;
  c += c2 + ((s - (t - b)) + (s2 - b));
  s = t;
}

// Partial sums of one thread's part of a tile: sums held as s + c pairs.
struct TileSums {
  float fn_s = 0.0f, fn_c = 0.0f;   // ||S_new||^2
  float fd_s = 0.0f, fd_c = 0.0f;   // ||S_old - X||^2
  float tr = 0.0f;                  // diagonal of S_new (at most one element per thread)
  bool bad = false;                 // a non-finite X
};

// 32 bytes to a 32-byte aligned address (one store instruction)
__device__ __forceinline__ void store32(void* p, const uint32_t (&v)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}

// Rolled tile epilogue of one thread: its row r (lane = row of the warp's 32),
// columns c0 .. c0 + 16 NG - 1 of a tile, whose sums the caller has written to
// tensor memory at ta_sum.  Forms S_new = sigma X + (1 - sigma) S_old
// (Eq. (eq:Sn) / Eq. (dB)), its FP16/BF16 hi/lo split (Sec. II C), the partial
// sums and stores each owned element (column >= row).  `release` is called
// when the sums have been read from tensor memory.
//
// Sixteen columns at a time; a warp's group of 16 columns lies above its 32
// rows (every element owned: the packed path), below them (nothing to do) or
// across the diagonal (two groups, the 32 x 32 block at the warp's rows).
//
// Memory access pattern.  A warp holds 32 consecutive rows (one per lane) and
// the same columns, so an access down a column (lane = row) is one contiguous
// segment while an access along the rows touches 32 lines.
//  * The FP32 master is kept in one orientation only: element (r, c),
//    c >= r, at (c, r) (the lower triangle with the diagonal), written and
//    read down the columns.  S_old[r][c] is read there; the next 16 columns
//    are loaded while the current ones are stored.  The readers of a whole
//    master (outputs, checkpoint reloads) take element (r, c) from
//    (max(r, c), min(r, c)).
//  * The 16-bit operand copies, which the tensor maps read as row panels,
//    are stored in both orientations.  Along the rows each lane stores its
//    16 columns as one whole 32-byte sector.  Down the columns two lanes
//    exchange halves so that each stores two rows of one column as a word.
// What bounds it: the instructions of the eight epilogue warps (about 9 K
// clocks per 128 x 256 part of a tile) and its stores (384 KB, 12 K clocks at
// the 32 B per clock an SM writes), which overlap in part.  With scalar
// arithmetic, 16-bit mirror stores, a shared-memory transpose for the rows and
// an FP64 tree for the partial sums a layer of n = 1000, k = 2 took 57 us and
// one of n = 2048, k = 3 157 us; now 51 and 149 us.  Sixteen warps of half the
// columns, or loads of S_old two groups ahead, do not change it.
//
// First 16-column group of a warp (rows from r0, columns from c0) that holds
// an owned element; its S_old values (element (c, r) at Sc + (c - c0) np).
__device__ __forceinline__ int epi_first_group(int r0, int c0) {
  return r0 > c0 ? (r0 - c0) >> 4 : 0;
}
// Groups of a warp's columns from c0 that lie left of column cend.
template <int NG>
__device__ __forceinline__ int epi_groups(int c0, int cend) {
  const int g = (cend - c0) >> 4;
  return g < NG ? g : NG;
}
__device__ __forceinline__ void epi_load_old(float (&olds)[16], const float* Sc, int np, int g16) {
#pragma unroll
  for (int q = 0; q < 16; ++q) olds[q] = __ldcg(Sc + (16 * g16 + q) * np);
}

// The calling epilogue warp's scratch block, after the partial sums at `red`.
__device__ __forceinline__ uint16_t* epi_block(float* red) {
  return reinterpret_cast<uint16_t*>(red + EPI_SUMS / 4) +
         ((threadIdx.x >> 5) - EPI_WARP0) * (32 * DLD);
}

// PRE: `olds` holds the first group's S_old on entry (read while the products
// still ran: tiles of up to 128 columns have the registers); dbuf: this warp's
// 32 x 32 block of scratch.
template <class CV, int NG, bool PRE, class Rel>
__device__ __forceinline__ void rolled_tile_epilogue(
    const uint32_t ta_sum, const float* __restrict__ Sold, float* Snew, typename CV::T* hi_new,
    typename CV::T* lo_new, const int lane, const int64_t Np, const int r, const int c0,
    const int cend, const float sg, const float om, const float scale_new, const bool write,
    float (&olds)[16], uint16_t* dbuf, TileSums& ts, Rel release) {
  const int r0 = r - lane;   // row of lane 0
  const int np = (int)Np;
  // groups below the warp's rows come first, groups above them last
  int g16 = epi_first_group(r0, c0);
  const int ng = epi_groups<NG>(c0, cend);
  if (g16 >= ng) {
    release();
    return;
  }
  // element (c, r) of the tile's columns at (c - c0) * np past col_base
  const size_t col_base = (size_t)c0 * Np + r;
  const size_t row_base = (size_t)r * Np + c0;
  const float* Sc = Sold + col_base;
  float* Snc = Snew + col_base;
  uint16_t* hic = reinterpret_cast<uint16_t*>(hi_new) + col_base;
  uint16_t* loc = reinterpret_cast<uint16_t*>(lo_new) + col_base;
  uint16_t* hir = reinterpret_cast<uint16_t*>(hi_new) + row_base;
  uint16_t* lor = reinterpret_cast<uint16_t*>(lo_new) + row_base;
  // column pairs: even lanes store (rows r, r + 1) of the even column, odd
  // lanes (rows r - 1, r) of the odd one
  const int odd = lane & 1;
  const uint32_t sel = odd ? 0x3276u : 0x5410u;
  uint16_t* hip = hic + (odd ? np - 1 : 0);
  uint16_t* lop = loc + (odd ? np - 1 : 0);
  const f32x2 sg2 = pack2(sg, sg), om2 = pack2(om, om), sc2 = pack2(scale_new, scale_new);
  const f32x2 neg2 = pack2(-1.0f, -1.0f), zero2 = pack2(0.0f, 0.0f);
  f32x2 fs = zero2, fc = zero2, fd = zero2, z = zero2;
  if constexpr (!PRE) epi_load_old(olds, Sc, np, g16);
#pragma unroll 1
  for (; g16 < ng; ++g16) {
    uint32_t xs[16];
    tmem_ld16(ta_sum + 16 * g16, xs);
    if (g16 == ng - 1) release();
    const int d = c0 + 16 * g16 - r0;   // < 32: a group on the diagonal
    if (d < 32) {
      // elements below the diagonal belong to their mirror elements; the one on
      // it counts half (the sums are doubled at the end)
      float xd = 0.0f, od = 0.0f;
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        if (d + e == lane) {
          xd = __uint_as_float(xs[e]);
          od = olds[e];
        }
        if (d + e < lane) xs[e] = 0u;
        if (d + e < lane) olds[e] = 0.0f;
      }
      const float dd = od - xd, n1 = sg * xd + om * od;
      ts.fd_s = fmaf(-0.5f * dd, dd, ts.fd_s);
      const float p = -0.5f * n1 * n1;
      ff_add(ts.fn_s, ts.fn_c, p, fmaf(-0.5f * n1, n1, -p));
      if (write) ts.tr += n1;
    }
    uint32_t hp[8], lp[8];   // hi / lo of the column pairs
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const f32x2 x = pack2(__uint_as_float(xs[2 * i]), __uint_as_float(xs[2 * i + 1]));
      const f32x2 o = pack2(olds[2 * i], olds[2 * i + 1]);
      z = fma2(x, zero2, z);               // becomes NaN with a non-finite x
      const f32x2 dx = fma2(x, neg2, o);
      fd = fma2(dx, dx, fd);               // each element counts twice: at the end
      const f32x2 nw = fma2(sg2, x, mul2(om2, o));
      // ||S_new||^2: the square as p + e (p = -np2), fs + p by TwoSum
      const f32x2 np2 = mul2(nw, mul2(nw, neg2));
      const f32x2 e = fma2(nw, nw, np2);
      const f32x2 tt = fma2(np2, neg2, fs);
      const f32x2 bp = fma2(fs, neg2, tt);
      const f32x2 t2 = fma2(fma2(bp, neg2, tt), neg2, fs);
      const f32x2 t3 = add2(np2, bp);
      fc = add2(fc, add2(fma2(t3, neg2, t2), e));
      fs = tt;
      const f32x2 y = mul2(nw, sc2);
      float y0, y1, n0, n1;
      unpack2(y, y0, y1);
      unpack2(nw, n0, n1);
      float h0, h1;
      hp[i] = CV::pack(y0, y1);
      CV::unpack(hp[i], h0, h1);
      float l0, l1;
      unpack2(fma2(pack2(h0, h1), neg2, y), l0, l1);
      lp[i] = CV::pack(l0, l1);
      if (write) {
        const int m = (16 * g16 + 2 * i) * np;
        if (d >= 32) {
          Snc[m] = n0;
          Snc[m + np] = n1;
          const uint32_t ho = __shfl_xor_sync(0xffffffffu, hp[i], 1);
          const uint32_t lo = __shfl_xor_sync(0xffffffffu, lp[i], 1);
          *reinterpret_cast<uint32_t*>(hip + m) = __byte_perm(hp[i], ho, sel);
          *reinterpret_cast<uint32_t*>(lop + m) = __byte_perm(lp[i], lo, sel);
        } else {
          if (d + 2 * i >= lane) Snc[m] = n0;
          if (d + 2 * i + 1 >= lane) Snc[m + np] = n1;
        }
      }
    }
    if (write) {
      if (d >= 32) {
        store32(hir + 16 * g16, hp);
        store32(lor + 16 * g16, lp);
      } else {
        // Both triangles of the 32 x 32 block on the diagonal (r0 and c0 are
        // multiples of 32) go through the warp's scratch block, whose finished
        // rows are stored whole: after the first group columns 0 .. 15 of rows
        // 0 .. 15, after the second the rest.  (Stored one by one, 16-bit
        // elements of every row went to 32 lines per instruction: 6.2 us of
        // epilogue in the layers of n = 128.)
#pragma unroll
        for (int part = 0; part < 2; ++part) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const uint32_t v = part ? lp[i] : hp[i];
            const int cl = d + 2 * i;   // column within the block
            if (cl >= lane) {
              dbuf[lane * DLD + cl] = (uint16_t)v;
              dbuf[cl * DLD + lane] = (uint16_t)v;
            }
            if (cl + 1 >= lane) {
              dbuf[lane * DLD + cl + 1] = (uint16_t)(v >> 16);
              dbuf[(cl + 1) * DLD + lane] = (uint16_t)(v >> 16);
            }
          }
          __syncwarp();
          // the columns left of this group belong to the block as well in the
          // second group's new rows (lanes 16 .. 31)
          uint16_t* row = (part ? lor : hir) + 16 * g16;
          const uint32_t* src = reinterpret_cast<const uint32_t*>(dbuf + lane * DLD + d);
          if (d == 16 || lane < 16) {
            uint32_t v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = src[i];
            store32(row, v);
          }
          if (d == 16 && lane >= 16) {
            uint32_t v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = src[i - 8];
            store32(row - 16, v);
          }
          __syncwarp();
        }
      }
    }
    if (g16 < ng - 1) epi_load_old(olds, Sc, np, g16 + 1);
  }
  float a0, a1, b0, b1;
  unpack2(fs, a0, a1);
  unpack2(fc, b0, b1);
  ff_add(ts.fn_s, ts.fn_c, a0, b0);
  ff_add(ts.fn_s, ts.fn_c, a1, b1);
  unpack2(fd, a0, a1);
  ff_add(ts.fd_s, ts.fd_c, a0, 0.0f);
  ff_add(ts.fd_s, ts.fd_c, a1, 0.0f);
  unpack2(z, a0, a1);
  ts.bad = ts.bad || !(a0 == 0.0f) || !(a1 == 0.0f);
}

// Partial sums of a CTA's part of a tile: each epilogue warp adds its lanes'
// sums as s + c pairs and leaves them in `red` (two buffers, used by
// successive items in turn); after one barrier the warp whose turn it is
// (`seq` mod EPI_WARPS) adds the eight warps in FP64 and writes the entry,
// while the others go on.  (Every thread's sums through an FP64 tree in
// shared memory took ten barriers and about 5 K clocks per item.)
constexpr int RED_FLOATS = 8;   // per warp: fn (s, c), fd (s, c), tr (s, c), bad, -
static_assert(2 * EPI_WARPS * RED_FLOATS * 4 <= EPI_SUMS, "two buffers");
__device__ __forceinline__ void tile_sums_out(TileSums ts, float* red, uint32_t seq, int ewarp,
                                              int lane, double* entry) {
  float tc = 0.0f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float ns = __shfl_down_sync(0xffffffffu, ts.fn_s, o);
    const float nc = __shfl_down_sync(0xffffffffu, ts.fn_c, o);
    const float ds = __shfl_down_sync(0xffffffffu, ts.fd_s, o);
    const float dc = __shfl_down_sync(0xffffffffu, ts.fd_c, o);
    const float t2 = __shfl_down_sync(0xffffffffu, ts.tr, o);
    const float tc2 = __shfl_down_sync(0xffffffffu, tc, o);
    ff_add(ts.fn_s, ts.fn_c, ns, nc);
    ff_add(ts.fd_s, ts.fd_c, ds, dc);
    ff_add(ts.tr, tc, t2, tc2);
  }
  const bool bad = __any_sync(0xffffffffu, ts.bad);
  float* buf = red + (seq & 1u) * EPI_WARPS * RED_FLOATS;
  if (lane == 0) {
    float4* p = reinterpret_cast<float4*>(buf + ewarp * RED_FLOATS);
    p[0] = make_float4(ts.fn_s, ts.fn_c, ts.fd_s, ts.fd_c);
    p[1] = make_float4(ts.tr, tc, bad ? 1.0f : 0.0f, 0.0f);
  }
  epi_sync();
  if (ewarp != (int)(seq % EPI_WARPS)) return;
  // lane 4 w + q: quantity q of warp w (trace, fro_new, fro_diff, bad)
  const int q = lane & 3, w = lane >> 2;
  const float* p = buf + w * RED_FLOATS;
  double v = q == 0 ? (double)p[4] + (double)p[5]
                    : (q == 1 ? (double)p[0] + (double)p[1]
                              : (q == 2 ? (double)p[2] + (double)p[3] : (double)p[6]));
#pragma unroll
  for (int o = 16; o >= 4; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  // elements off the diagonal count twice (and those on it were halved)
  if (lane < 4) entry[lane] = (lane == kQFroNew || lane == kQFroDiff) ? 2.0 * v : v;
}
static_assert(kQTrace == 0 && kQFroNew == 1 && kQFroDiff == 2 && kQBad == 3 && EPI_WARPS == 8,
              "lanes of tile_sums_out");

template <bool BF16>
__global__ void __launch_bounds__(NUM_THREADS, 1)
    layer_tc_kernel(const __grid_constant__ CUtensorMap mapA,
                    const __grid_constant__ CUtensorMap mapB, State* st,
                    float* __restrict__ master, uint16_t* __restrict__ ops, int64_t Np, int k,
                    double* __restrict__ partials, int64_t ptiles, uint64_t limit_ns, int chunk,
                    int inject_stall) {
  using CV = Cvt<BF16>;
  using H16 = typename CV::T;
  extern __shared__ uint8_t smem_raw[];
  if (st->done) return;

  // ---- plan of this layer (identical in every CTA)
  uint32_t jmask = st->plan_square ? 1u : 0u;
  for (int j = 0; j < k; ++j)
    if (st->plan_resp[j]) jmask |= 1u << (1 + j);
  const int njobs = __popc(jmask);
  if (njobs == 0) return;
  const int cur0 = st->cur0;
  const int sigma = st->sigma_cur;
  const int write0 = st->plan_write0;
  const int s0e = st->s0_exp;
  const int z0c = st->z0_cur, z0n = st->z0_next;
  const int k1 = st->order >= 2 ? st->k1 : k;   // first-order directions

  const int64_t tiles = num_tiles(Np);
  const int64_t items = tiles * njobs;
  const int kblocks = k_blocks(st->n);

  // ---- shared memory carve-up (1024-aligned stage ring)
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - raw);
  const uint32_t ring = base;
  uint8_t* misc = gbase + STAGES * STAGE_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(misc);  // full, empty, tfull, tempty, drain
  const uint32_t bar_full = smem_u32(bars);
  const uint32_t bar_empty = bar_full + 8 * STAGES;
  const uint32_t bar_tfull = bar_empty + 8 * STAGES;
  const uint32_t bar_tempty = bar_tfull + 8 * 2;
  const uint32_t bar_drain = bar_tempty + 8 * 2;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(misc + 128);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 136);
  float* red = reinterpret_cast<float*>(misc + 1024);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(bar_full + 8 * s, 1);
      mbar_init(bar_empty + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar_tfull + 8 * b, 1);
      mbar_init(bar_tempty + 8 * b, EPI_WARPS);  // one arrive per epilogue warp
    }
    mbar_init(bar_drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32((const void*)tmem_slot)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem_base = *tmem_slot;
  int* timeout_global = &st->timeout_flag;

  if (warp == 0) {
    // ================= TMA producer =================
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      int inflight = 0;  // stages issued whose completion this thread has not observed
      bool ok = true;
      for (int64_t it = blockIdx.x; it < items && ok; it += gridDim.x) {
        const int job = job_at(jmask, (int)(it / tiles));
        int I, J;
        tile_coords(it % tiles, &I, &J);
        const int passes = job_passes(job, k1);
        for (int pass = 0; pass < passes && ok; ++pass) {
          // A = rows I of slot mA, B = rows J of slot mB (B[k][j] = B[j][k])
          int mA, mB;
          job_operands(job, pass, k1, &mA, &mB);
          const int bufA = mA == 0 ? cur0 : st->cur1[mA - 1];
          const int bufB = mB == 0 ? cur0 : st->cur1[mB - 1];
          const int zAh = zop(mA, bufA, 0, k, z0c), zAl = zop(mA, bufA, 1, k, z0c);
          const int zBh = zop(mB, bufB, 0, k, z0c), zBl = zop(mB, bufB, 1, k, z0c);
          for (int kb = 0; kb < kblocks; ++kb) {
            if (!mbar_wait(bar_empty + 8 * stage, phase ^ 1, limit_ns, abort_flag,
                           timeout_global)) {
              ok = false;
              break;
            }
            const uint32_t sA = ring + stage * STAGE_BYTES;
            const uint32_t fb = bar_full + 8 * stage;
            mbar_expect_tx(fb, STAGE_BYTES);
            tma_load_3d(sA, &mapA, kb * BK, I * BM, zAh, fb);
            tma_load_3d(sA + A_BYTES, &mapA, kb * BK, I * BM, zAl, fb);
            tma_load_3d(sA + 2 * A_BYTES, &mapB, kb * BK, J * BN, zBh, fb);
            tma_load_3d(sA + 2 * A_BYTES + B_BYTES, &mapB, kb * BK, J * BN, zBl, fb);
            inflight = inflight < STAGES ? inflight + 1 : STAGES;
            if (++stage == STAGES) {
              stage = 0;
              phase ^= 1;
            }
          }
        }
      }
      if (!ok) {
        // drain: wait (bounded) until the copies already issued have landed
        int s = stage;
        uint32_t ph = phase;
        for (int i = 0; i < inflight; ++i) {
          if (--s < 0) {
            s = STAGES - 1;
            ph ^= 1;
          }
          const uint64_t t0 = gtimer();
          while (!mbar_try_wait(bar_full + 8 * s, ph) && gtimer() - t0 < limit_ns) {
          }
        }
      }
    }
  } else if (warp == 1) {
    // ================= MMA issuer =================
    // The K sequence of an item (all passes) is cut into chunks of `chunk`
    // stages; each chunk accumulates from zero into one of the two TMEM
    // accumulators and is summed by the epilogue in FP32 on the CUDA cores.
    if (lane == 0) {
      constexpr uint32_t idesc = make_idesc(BF16 ? 1 : 0);
      int stage = 0;
      uint32_t phase = 0;
      int ab = 0;
      uint32_t abphase = 0;
      // test hook: wait on a barrier nothing arrives on, so that the bounded
      // waits of every role run out and the timeout path is exercised
      bool ok = !(inject_stall &&
                  !mbar_wait(bar_drain, 0, limit_ns, abort_flag, timeout_global));
      for (int64_t it = blockIdx.x; it < items && ok; it += gridDim.x) {
        const int job = job_at(jmask, (int)(it / tiles));
        const int nst = job_passes(job, k1) * kblocks;
        uint32_t d = 0, acc = 0;
        int sp = 0;   // stage within its K pass
        int cp = 0;   // stage within its accumulation chunk
        for (int si = 0; si < nst; ++si) {
          if (cp == 0) {
            if (!mbar_wait(bar_tempty + 8 * ab, abphase ^ 1, limit_ns, abort_flag,
                           timeout_global)) {
              ok = false;
              break;
            }
            fence_after();
            d = tmem_base + (uint32_t)(ab * BN);
            acc = 0;
          }
          if (!mbar_wait(bar_full + 8 * stage, phase, limit_ns, abort_flag, timeout_global)) {
            ok = false;
            break;
          }
          fence_after();
          const uint32_t sA = ring + stage * STAGE_BYTES;
          const uint64_t ah = sw64_desc(sA), al = sw64_desc(sA + A_BYTES);
          const uint64_t bh = sw64_desc(sA + 2 * A_BYTES);
          const uint64_t bl = sw64_desc(sA + 2 * A_BYTES + B_BYTES);
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk) {
            const uint64_t off = (uint64_t)((kk * 32) >> 4);  // 16 elements = 32 B
            mma_f16(d, ah + off, bh + off, idesc, acc);        // hi * hi
            acc = 1;
            mma_f16(d, ah + off, bl + off, idesc, 1);          // hi * lo
            mma_f16(d, al + off, bh + off, idesc, 1);          // lo * hi
          }
          mma_commit(bar_empty + 8 * stage);  // frees the stage when these MMAs finish
          if (++stage == STAGES) {
            stage = 0;
            phase ^= 1;
          }
          const bool chunk_end = cp == chunk - 1 || sp == kblocks - 1;
          if (++cp == chunk || sp == kblocks - 1) cp = 0;
          if (++sp == kblocks) sp = 0;
          if (chunk_end) {
            mma_commit(bar_tfull + 8 * ab);  // chunk accumulator ready
            if (++ab == 2) {
              ab = 0;
              abphase ^= 1;
            }
          }
        }
      }
      // wait (bounded) until every MMA this thread issued has completed, so
      // TMEM is idle before it is freed
      mma_commit(bar_drain);
      const uint64_t t0 = gtimer();
      while (!mbar_try_wait(bar_drain, 0) && gtimer() - t0 < limit_ns) {
      }
    }
  } else if (warp >= EPI_WARP0) {
    // ================= epilogue (warps 2..9) =================
    // Thread = one row of the tile (TMEM lane) and one half of its columns.
    const int q = warp & 3;                 // TMEM lane quadrant of this warp
    const int half = (warp - EPI_WARP0) >> 2;  // column half: 0 -> 0..127, 1 -> 128..255
    const int rloc = 32 * q + lane;         // row within the tile
    const size_t mat = (size_t)Np * Np;
    const uint32_t tlane = (uint32_t)(32 * q) << 16;
    int ab = 0;
    uint32_t abphase = 0;
    bool alive = true;
    uint32_t seq = 0;   // items done (tile_sums_out)
    const bool crev = false;   // this kernel always runs the passes forwards
    for (int64_t it = blockIdx.x; it < items && alive; it += gridDim.x) {
      const int job = job_at(jmask, (int)(it / tiles));
      const int passes = job_passes(job, k1);
      const int cpp = (kblocks + chunk - 1) / chunk;   // chunks per pass
      const int nchunks = passes * cpp;
      // exact power-of-two unscale of the products of passes 0 and 1
      // (passes >= 2 of higher-order terms: cross_unscale)
      const float u01 = ldexpf(1.0f, -(s0e + (job == 0 ? s0e : st->s1_exp_cur[job - 1])));

      // ---- sum the chunk accumulators in FP32 (round to nearest)
      float sum[128];
#pragma unroll
      for (int i = 0; i < 128; ++i) sum[i] = 0.0f;
      for (int ch = 0; ch < nchunks; ++ch) {
        const bool ok =
            mbar_wait(bar_tfull + 8 * ab, abphase, limit_ns, abort_flag, timeout_global);
        // all epilogue threads take the same branch (warp-collective
        // tcgen05.ld follows)
        if (!epi_all(ok && !*abort_flag)) {
          alive = false;
          break;
        }
        fence_after();
        const uint32_t ta = tmem_base + tlane + (uint32_t)(ab * BN + half * 128);
        const int pc = chunk_pass(ch, cpp, passes, crev);
        const float u = pc < 2 ? u01 : cross_unscale(st, job, pc, k1);
#pragma unroll
        for (int cc = 0; cc < 8; ++cc) {
          uint32_t x[16];
          tmem_ld16(ta + 16 * cc, x);
#pragma unroll
          for (int i = 0; i < 16; ++i)
            sum[16 * cc + i] = fmaf(__uint_as_float(x[i]), u, sum[16 * cc + i]);
        }
        if (ch + 1 == nchunks) break;   // keep the last chunk's buffer
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_tempty + 8 * ab);
        if (++ab == 2) {
          ab = 0;
          abphase ^= 1;
        }
      }
      if (!alive) break;
      // the tile's sums go back into its last chunk's buffer
      const uint32_t ta_sum = tmem_base + tlane + (uint32_t)(ab * BN + half * 128);
#pragma unroll
      for (int cc = 0; cc < 8; ++cc) tmem_st16(ta_sum + 16 * cc, sum + 16 * cc);
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");

      // ---- fused layer update, split and stores
      const int64_t t = it % tiles;
      int I, J;
      tile_coords(t, &I, &J);
      const int curj = job == 0 ? cur0 : st->cur1[job - 1];
      const int e_new = job == 0 ? s0e : st->s1_exp_next[job - 1];
      const float scale_new = ldexpf(1.0f, e_new);   // exact power of two
      const float sg = (float)sigma, om = 1.0f - (float)sigma;
      const bool write = job != 0 || write0;
      const int r = I * BM + rloc;
      const int c0 = J * BN + half * 128;
      const float* Sold = master + (size_t)(curj * (1 + k) + job) * mat;
      float* Snew = master + (size_t)((curj ^ 1) * (1 + k) + job) * mat;
      const int zh_new = job == 0 ? z0n : zslice(curj ^ 1, job, 0, k);
      H16* hi_new = reinterpret_cast<H16*>(ops) + (size_t)zh_new * mat;
      H16* lo_new = reinterpret_cast<H16*>(ops) + (size_t)(zh_new + 1) * mat;

      float olds[16];
      TileSums ts;
      auto release = [&]() {   // the accumulator goes back to the MMA
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_tempty + 8 * ab);
      };
      rolled_tile_epilogue<CV, 8, false>(ta_sum, Sold, Snew, hi_new, lo_new, lane, Np, r, c0,
                                         kblocks * BK, sg, om, scale_new, write, olds,
                                         epi_block(red), ts, release);
      if (++ab == 2) {
        ab = 0;
        abphase ^= 1;
      }
      tile_sums_out(ts, red, seq++, warp - EPI_WARP0, lane,
                    partials + ((size_t)job * ptiles + t) * kNQ);
    }
  }

  // ---- teardown: everyone done (or aborted); free TMEM
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                 "r"(TMEM_COLS));
  }
}

// ---------------------------------------------------------------------------
// CTA-pair variant (cta_group::2).  A cluster of two CTAs computes a
// 256 x 256 tile: CTA r holds rows 128 r .. 128 r + 127 of A and B rows
// (output columns) 128 r .. 128 r + 127; the leader (rank 0) issues
// M = 256, N = 256 MMAs that read A from each CTA's own shared memory and B
// from both, and each CTA's tensor memory receives its 128 rows of the
// accumulator.  Per SM this cuts the operand bytes loaded for 32 columns of K
// and 256 columns of the tile from 48 to 32 KB.
//   full[s]   leader only: leader producer's expect_tx of both CTAs' stages;
//             both CTAs' TMA loads complete their bytes on it
//   empty[s]  each CTA: the leader's MMA commit arrives on both (multicast)
//   tfull[b]  each CTA: leader's commit, multicast
//   tempty[b] leader only: 16 arrivals (8 epilogue warps per CTA)

static_assert(272 + 4 * kHeadWords <= 1024, "the control block's head below the partial sums");

// Geometry of the pair kernels' tiles, 256 rows x NT columns: each CTA loads
// its 128 A rows and NT / 2 B rows, SK columns wide, per stage, and tensor
// memory holds ACC accumulators of NT columns.  A stage is one 128-byte swizzle
// span of K: with 64-byte rows and stages of 32 columns the 256 x 256 tiles
// waited for operands (n = 8192 k = 3 solve 295.7 ms, now 290.7; n = 4096
// k = 1 layer 432 -> 411 us).
template <int NT>
struct PairTile {
  static constexpr int SK = 64;                                 // K elements per stage
  static constexpr int B_ROWS = NT / 2;
  static constexpr int PA_BYTES = BM * SK * 2;
  static constexpr int PB_BYTES = B_ROWS * SK * 2;
  static constexpr int STAGE = 2 * PA_BYTES + 2 * PB_BYTES;     // 64, 48, 40 KB
  static constexpr int STAGES = 200 * 1024 / STAGE;             // 3, 4, 5
  static constexpr int ACC = NT == 256 ? 2 : 4;
  static constexpr int COLS = ACC * NT;                         // tensor-memory columns
  static constexpr int SPLIT = BN / NT;                         // tiles per 256 x 256 tile
  static constexpr int SMEM = STAGES * STAGE + 1024 + 1024 + EPI_SCRATCH;
  static_assert(8 * (2 * STAGES + 2 * ACC + 1) <= 256, "barriers below the TMEM slot");
};

__host__ __device__ inline int64_t num_pair_tiles(int64_t Np) {
  const int64_t tj = Np / BN;
  return tj * (tj + 1) / 2;
}
// pair tile t -> (I2, J), I2 <= J, J-major
__device__ __forceinline__ void pair_tile_coords(unsigned t, int* I2, int* J) {
  unsigned j = (unsigned)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while ((j + 1) * (j + 2) / 2 <= t) ++j;
  while (j * (j + 1) / 2 > t) --j;
  *J = (int)j;
  *I2 = (int)(t - j * (j + 1) / 2);
}

// Banded order of the pair tiles (I2 <= J): column blocks are grouped into
// bands of `band` blocks; inside a band the tiles run I2-major, so the pairs
// working at the same time cover a compact block of rows and columns and
// share their operand panels in L2.  band <= 0 keeps the plain J-major order.
// (Tile indexes fit 32 bits: a matrix of 2^31 tiles would not fit any memory.)
__device__ __forceinline__ void pair_tile_banded(unsigned t, int tj, int band, int* I2, int* J) {
  if (band <= 0) {
    pair_tile_coords(t, I2, J);
    return;
  }
  unsigned J0 = 0;
  while (true) {
    const unsigned w = tj - J0 < (unsigned)band ? tj - J0 : band;
    const unsigned cnt = J0 * w + w * (w + 1) / 2;   // tiles in this band
    if (t < cnt || J0 + w >= (unsigned)tj) {
      if (t < J0 * w) {          // rows above the band's diagonal block
        *I2 = (int)(t / w);
        *J = (int)(J0 + t % w);
        return;
      }
      unsigned u = t - J0 * w;    // upper triangle of the w x w diagonal block
      unsigned r = 0;
      while (u >= w - r) {
        u -= w - r;
        ++r;
      }
      *I2 = (int)(J0 + r);
      *J = (int)(J0 + r + u);
      return;
    }
    t -= cnt;
    J0 += w;
  }
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank) {
  uint32_t out;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"(addr), "r"(rank));
  return out;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}
// Arrive on a barrier of another CTA of the cluster.  Release at CTA scope
// only: the arrival signals that this warp's tensor-memory reads are done
// (tcgen05.wait::ld has returned), not that its global stores are visible,
// so no cluster-scope fence (which would wait for the previous tile's
// stores) is needed.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* map, int x, int y,
                                                 int z, uint32_t leader_bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(leader_bar)
      : "memory");
}
__device__ __forceinline__ void mma_f16_pair(uint32_t d_tmem, uint64_t a, uint64_t b,
                                             uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}
__device__ __forceinline__ void mma_commit_pair(uint32_t bar) {
  const uint16_t mask = 0x3;
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
      " [%0], %1;" ::"r"(bar), "h"(mask)
      : "memory");
}
__host__ __device__ constexpr uint32_t make_idesc_m256(int ab_type, int n) {
  return (1u << 4) | ((uint32_t)ab_type << 7) | ((uint32_t)ab_type << 10) |
         ((uint32_t)(n >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
}

// Position in the shared-memory stage ring (stage index and phase bit) or
// in the two tensor-memory accumulators (buffer and phase bit).
struct RingPos {
  int idx = 0;
  uint32_t phase = 0;
  __device__ __forceinline__ void next(int size) {
    if (++idx == size) {
      idx = 0;
      phase ^= 1;
    }
  }
};

// TMA producer of a pair kernel, one work item: the item's passes over its
// K blocks (backwards when `rev`), each stage the hi and lo halves of this
// CTA's A rows (128-row map) and B rows (NT / 2-row map), signalled on the
// pair leader's full barrier.  False when a bounded wait expired or the CTA
// aborted.
template <int NT>
__device__ __forceinline__ bool produce_item(
    RingPos& rg, const CUtensorMap* map, const CUtensorMap* mapB, const State* st, int job,
    int passes, int k, int k1, int cur0, int z0c, int rowA, int rowB, int kblocks, bool rev,
    bool leader, uint32_t ring, uint32_t bar_full, uint32_t bar_empty, uint32_t lead_full,
    uint64_t limit_ns, volatile int* abort_flag, int* timeout_global) {
  using PT = PairTile<NT>;
  for (int pp = 0; pp < passes; ++pp) {
    const int pass = rev ? passes - 1 - pp : pp;
    int mA, mB;
    job_operands(job, pass, k1, &mA, &mB);
    const int bufA = mA == 0 ? cur0 : st->cur1[mA - 1];
    const int bufB = mB == 0 ? cur0 : st->cur1[mB - 1];
    const int zAh = zop(mA, bufA, 0, k, z0c), zAl = zop(mA, bufA, 1, k, z0c);
    const int zBh = zop(mB, bufB, 0, k, z0c), zBl = zop(mB, bufB, 1, k, z0c);
    const int nst = (kblocks * BK + PT::SK - 1) / PT::SK;
    for (int kq = 0; kq < nst; ++kq) {
      const int x = (rev ? nst - 1 - kq : kq) * PT::SK;
      if (!mbar_wait_warp(bar_empty + 8 * rg.idx, rg.phase ^ 1, limit_ns, abort_flag,
                          timeout_global))
        return false;
      const uint32_t sA = ring + rg.idx * PT::STAGE;
      const uint32_t fb = lead_full + 8 * rg.idx;
      if (elect_one()) {
        if (leader) mbar_expect_tx(bar_full + 8 * rg.idx, 2 * PT::STAGE);
        tma_load_3d_pair(sA, map, x, rowA, zAh, fb);
        tma_load_3d_pair(sA + PT::PA_BYTES, map, x, rowA, zAl, fb);
        tma_load_3d_pair(sA + 2 * PT::PA_BYTES, mapB, x, rowB, zBh, fb);
        tma_load_3d_pair(sA + 2 * PT::PA_BYTES + PT::PB_BYTES, mapB, x, rowB, zBl, fb);
      }
      __syncwarp();
      rg.next(PT::STAGES);
    }
  }
  return true;
}

// Before a CTA exits, wait (bounded) for the copies it issued to land: the
// last `stages` stages were released by MMA commits or are pending.
__device__ __forceinline__ void producer_drain(RingPos rg, int stages, uint32_t bar_empty,
                                               uint64_t limit_ns) {
  for (int i = 0; i < stages; ++i) {
    const uint64_t t0 = gtimer();
    while (!mbar_try_wait(bar_empty + 8 * rg.idx, rg.phase ^ 1) && gtimer() - t0 < limit_ns) {
    }
    rg.next(stages);
  }
}

// MMA issuer of a pair kernel (leader CTA, one warp), one work item: per K
// block of 32 the three products hi*hi, hi*lo, lo*hi for two K16 steps into
// the current accumulation chunk; a chunk ends every `chunk` blocks and at the
// end of each K pass (so chunks never straddle a pass), the first of a pass
// after chunk - cp0 blocks, and is then published to both CTAs.  cols: the
// tile's columns (a multiple of 32).  False when a bounded wait expired.
//
// The whole warp runs the loop and one elected lane issues: what bounds a
// narrow tile is the issue of its MMAs, and with the loop under `lane == 0`
// the compiler handles each instruction's operands per lane.  Per 32-wide
// block at N = 64 / 128 that took 0.39 / 0.41 us, with the elected lane 0.24 us
// each.
template <bool BF16, int NT>
__device__ __forceinline__ bool mma_item(RingPos& rg, RingPos& tb, int passes, int kblocks,
                                         int chunk, int cp0, bool rev, int cols,
                                         uint32_t tmem_base, uint32_t ring, uint32_t bar_full,
                                         uint32_t bar_empty, uint32_t bar_tfull,
                                         uint32_t bar_tempty, uint64_t limit_ns,
                                         volatile int* abort_flag, int* timeout_global) {
  using PT = PairTile<NT>;
  const uint32_t idesc = make_idesc_m256(BF16 ? 1 : 0, cols);
  constexpr int H = PT::SK / BK;   // blocks per stage
  const int nst = (kblocks + H - 1) / H;
  for (int pass = 0; pass < passes; ++pass) {
    uint32_t d = 0;
    int cp = cp0;   // block within its accumulation chunk
    bool fresh = true;
    for (int sq = 0; sq < nst; ++sq) {
      if (!mbar_wait_warp(bar_full + 8 * rg.idx, rg.phase, limit_ns, abort_flag, timeout_global))
        return false;
      const uint32_t sA = ring + rg.idx * PT::STAGE;
      const uint64_t ah = sw128_desc(sA), al = sw128_desc(sA + PT::PA_BYTES);
      const uint64_t bh = sw128_desc(sA + 2 * PT::PA_BYTES);
      const uint64_t bl = sw128_desc(sA + 2 * PT::PA_BYTES + PT::PB_BYTES);
#pragma unroll
      for (int hq = 0; hq < H; ++hq) {
        const int h = rev ? H - 1 - hq : hq;
        const int blk = (rev ? nst - 1 - sq : sq) * H + h;
        if (blk >= kblocks) continue;   // the padding half of the last stage
        uint32_t acc = 1;
        if (fresh) {
          if (!mbar_wait_warp(bar_tempty + 8 * tb.idx, tb.phase ^ 1, limit_ns, abort_flag,
                              timeout_global))
            return false;
          d = tmem_base + (uint32_t)(tb.idx * NT);
          acc = 0;
        }
        fence_after();
        fresh = ++cp == chunk || blk == (rev ? 0 : kblocks - 1);   // the chunk's last block
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk) {
            const uint64_t off = (uint64_t)((h * BK * 2 + kk * 32) >> 4);
            mma_f16_pair(d, ah + off, bh + off, idesc, kk == 0 ? acc : 1u);   // hi * hi
            mma_f16_pair(d, ah + off, bl + off, idesc, 1);                    // hi * lo
            mma_f16_pair(d, al + off, bh + off, idesc, 1);                    // lo * hi
          }
          if (fresh) mma_commit_pair(bar_tfull + 8 * tb.idx);   // chunk ready in both CTAs
        }
        __syncwarp();
        if (fresh) {
          tb.next(PT::ACC);
          cp = 0;
        }
      }
      if (elect_one()) mma_commit_pair(bar_empty + 8 * rg.idx);   // frees the stage in both CTAs
      __syncwarp();
      rg.next(PT::STAGES);
    }
  }
  return true;
}

// Soft round alignment of the pair kernel's producers.  Items go to the
// pairs round-robin, so the 76 tiles of a round share their operand panels
// in L2 only while the pairs stay in step; a pair that drifts a round ahead
// fetches those panels from HBM again (with the fast, coalesced tile
// epilogue the pairs do drift, and DRAM reads per layer double).  The count
// is a scheduling hint only: no data depends on it.  At the start of each
// round r >= 1 a producer counts itself in and waits until every CTA that
// has an item in round r has started it.  The wait is bounded
// (kRoundAlignNs) and is never an error: after an expiry that producer stops
// waiting for the rest of the launch (it still counts itself in), so a grid
// whose CTAs are not all resident at once costs at most one bound.
constexpr uint64_t kRoundAlignNs = 300000;
__device__ __forceinline__ void round_start(unsigned* ctr, int64_t round, int64_t items,
                                            int64_t npairs, bool& align) {
  atomicAdd(ctr, 1u);
  if (!align) return;
  // CTAs with an item in rounds 1 .. round (only the last round is partial)
  const int64_t upto = (round + 1) * npairs < items ? (round + 1) * npairs : items;
  const unsigned target = (unsigned)(2 * (upto - npairs));
  const uint64_t t0 = gtimer();
  while (*reinterpret_cast<volatile unsigned*>(ctr) < target) {
    if (gtimer() - t0 > kRoundAlignNs) {
      align = false;
      return;
    }
    __nanosleep(128);
  }
}

// Tile epilogue of the pair kernel: after a tile's last chunk the sums are
// written back into that chunk's tensor-memory buffer and read 16 columns at
// a time by rolled_tile_epilogue (little code per tile; one register spilled at
// 256 columns, none below);
// the buffer returns to the MMA after that loop, so the MMA runs one chunk
// ahead of the epilogue during it.
template <bool BF16, int NT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(NUM_THREADS, 1)
    layer_tc2_kernel(const __grid_constant__ CUtensorMap mapA,
                     const __grid_constant__ CUtensorMap mapB, State* gst,
                     float* __restrict__ master, uint16_t* __restrict__ ops, int64_t Np, int k,
                     double* __restrict__ partials, int64_t ptiles, uint64_t limit_ns, int chunk,
                     int k_snake, int snake_pairs, int band, int inject_stall, int round_align) {
  using PT = PairTile<NT>;
  constexpr int SP = PT::SPLIT;
  using CV = Cvt<BF16>;
  using H16 = typename CV::T;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t rank = cluster_rank();
  const bool leader = rank == 0;
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - raw);
  const uint32_t ring = base;
  uint8_t* misc = gbase + PT::STAGES * PT::STAGE;
  uint64_t* bars = reinterpret_cast<uint64_t*>(misc);
  const uint32_t bar_full = smem_u32(bars);
  const uint32_t bar_empty = bar_full + 8 * PT::STAGES;
  const uint32_t bar_tfull = bar_empty + 8 * PT::STAGES;
  const uint32_t bar_tempty = bar_tfull + 8 * PT::ACC;
  const uint32_t bar_drain = bar_tempty + 8 * PT::ACC;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(misc + 256);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 264);
  float* red = reinterpret_cast<float*>(misc + 1024);
  const uint32_t lead_full = map_to_rank(bar_full, 0);
  const uint32_t lead_tempty = map_to_rank(bar_tempty, 0);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < PT::STAGES; ++s) {
      mbar_init(bar_full + 8 * s, 1);
      mbar_init(bar_empty + 8 * s, 1);
    }
    for (int b = 0; b < PT::ACC; ++b) {
      mbar_init(bar_tfull + 8 * b, 1);
      mbar_init(bar_tempty + 8 * b, 2 * EPI_WARPS);
    }
    mbar_init(bar_drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32((const void*)tmem_slot)),
                 "r"(PT::COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
  }
  if (warp == 0 && elect_one()) {
    prefetch_tensormap(&mapA);
    prefetch_tensormap(&mapB);
  }
  fence_before();
  cluster_sync_all();   // barriers of both CTAs initialised, TMEM allocated
  fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // ---- everything above ran while the previous kernels of the stream finished
  pdl_wait();
  pdl_launch();
  State* st = reinterpret_cast<State*>(misc + 272);   // the control block's head
  for (int i = threadIdx.x; i < kHeadWords; i += NUM_THREADS)
    reinterpret_cast<unsigned*>(st)[i] = __ldcg(reinterpret_cast<const unsigned*>(gst) + i);
  __syncthreads();

  // ---- plan of this layer (the same in every CTA)
  uint32_t jmask = 0;
  if (!st->done) {
    jmask = st->plan_square ? 1u : 0u;
    for (int j = 0; j < k; ++j)
      if (st->plan_resp[j]) jmask |= 1u << (1 + j);
  }
  const int njobs = __popc(jmask);
  const int cur0 = st->cur0;
  const int sigma = st->sigma_cur;
  const int write0 = st->plan_write0;
  const int s0e = st->s0_exp;
  const int z0c = st->z0_cur, z0n = st->z0_next;
  const int k1 = st->order >= 2 ? st->k1 : k;   // first-order directions
  // virtual index of the first item (0, except when the backward recomputes
  // a square alone: it then numbers the square's items as the forward launch
  // did, after its response items, so each tile keeps its round and K-snake
  // direction and the recomputed states are bit-identical)
  const unsigned vbase = SP * (unsigned)st->item_base;

  const unsigned pair = blockIdx.x >> 1;
  const unsigned npairs = gridDim.x >> 1;
  const unsigned tiles = (unsigned)num_pair_tiles(Np);
  const unsigned items = SP * tiles * (unsigned)njobs;
  const int kblocks = k_blocks(st->n);
  const int cend = kblocks * BK;

  int* timeout_global = &gst->timeout_flag;

  // All pairs move through their tiles' K ranges in near lockstep; in odd
  // rounds of the 256 x 256 tiles the sweep runs backwards (passes and K
  // blocks), so a round starts on the panel slices the previous round loaded
  // last, which are still in L2.  Narrower tiles keep the direction of the
  // 256 x 256 tile they are part of: an element's sums, and so the results,
  // are the same bit for bit at every width.
  auto item_rev = [&](unsigned v) {
    return k_snake && ((v / SP / (unsigned)snake_pairs) & 1u);
  };

  if (njobs == 0) {
    // nothing to do in this launch
  } else if (warp == 0) {
    // ================= TMA producer (both CTAs load their own halves) ======
    {
      RingPos rg;
      bool ok = true;
      bool align = round_align != 0 && SP == 1;
      for (unsigned v = pair; v < vbase + items && ok; v += npairs) {
        if (v < vbase) continue;
        const unsigned it = (v - vbase) / SP;
        if (SP == 1 && v >= npairs) {
          if (lane == 0) round_start(&gst->round_ctr, v / npairs, items, npairs, align);
          __syncwarp();
        }
        const int job = job_at(jmask, (int)(it / tiles));
        int I2, J;
        pair_tile_banded(it % tiles, (int)(Np / BN), band, &I2, &J);
        const int cb = J * BN + (int)(v % SP) * NT, cols = tile_cols(cb, NT, cend);
        if (SP > 1 && cols == 0) continue;
        ok = produce_item<NT>(rg, &mapA, &mapB, st, job, job_passes(job, k1), k, k1, cur0, z0c,
                              I2 * 2 * BM + (int)rank * BM, cb + (int)rank * (cols / 2), kblocks,
                              item_rev(v), leader, ring, bar_full, bar_empty, lead_full, limit_ns,
                              abort_flag, timeout_global);
      }
      if (lane == 0) producer_drain(rg, PT::STAGES, bar_empty, limit_ns);
    }
  } else if (warp == 1) {
    // ================= MMA issuer (leader CTA only) =================
    if (leader) {
      RingPos rg, tb;
      // test hook (see the single-CTA kernel)
      bool ok = !(inject_stall &&
                  !mbar_wait_warp(bar_drain, 0, limit_ns, abort_flag, timeout_global));
      for (unsigned v = pair; v < vbase + items && ok; v += npairs) {
        if (v < vbase) continue;
        const unsigned it = (v - vbase) / SP;
        const int job = job_at(jmask, (int)(it / tiles));
        int I2, J;
        pair_tile_banded(it % tiles, (int)(Np / BN), band, &I2, &J);
        const int cols = tile_cols(J * BN + (int)(v % SP) * NT, NT, cend);
        if (SP > 1 && cols == 0) continue;
        ok = mma_item<BF16, NT>(rg, tb, job_passes(job, k1), kblocks, chunk,
                                kchunk0(Np, kblocks, chunk, item_rev(v)), item_rev(v), cols,
                                tmem_base, ring,
                                bar_full, bar_empty, bar_tfull, bar_tempty, limit_ns, abort_flag,
                                timeout_global);
      }
      if (elect_one())
        asm volatile(
            "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                bar_drain)
            : "memory");
      __syncwarp();
      const uint64_t t0 = gtimer();
      while (!mbar_try_wait(bar_drain, 0) && gtimer() - t0 < limit_ns) {
      }
    }
  } else if (warp >= EPI_WARP0) {
    // ================= epilogue (both CTAs, own 128 rows) =================
    const int q = warp & 3;
    const int half = (warp - EPI_WARP0) >> 2;
    const int rloc = 32 * q + lane;
    const size_t mat = (size_t)Np * Np;
    const uint32_t tlane = (uint32_t)(32 * q) << 16;
    RingPos ab;
    bool alive = true;
    uint32_t seq = 0;   // items done (tile_sums_out)
    for (unsigned v = pair; v < vbase + items && alive; v += npairs) {
      if (v < vbase) continue;
      const unsigned it = (v - vbase) / SP;
      const bool crev = item_rev(v);
      const int job = job_at(jmask, (int)(it / tiles));
      const int passes = job_passes(job, k1);
      // chunks per pass
      const int cpp = (kchunk0(Np, kblocks, chunk, crev) + kblocks + chunk - 1) / chunk;
      const int nchunks = passes * cpp;
      // exact power-of-two unscale of the products of passes 0 and 1
      // (passes >= 2 of higher-order terms: cross_unscale)
      const float u01 = ldexpf(1.0f, -(s0e + (job == 0 ? s0e : st->s1_exp_cur[job - 1])));
      // S_old of this thread's first columns: narrow tiles have the registers to
      // read them while the products run
      float olds[16];
      if constexpr (NT < BN) {
        int I2, J;
        pair_tile_banded(it % tiles, (int)(Np / BN), band, &I2, &J);
        if (tile_cols(J * BN + (int)(v % SP) * NT, NT, cend) == 0) {   // nothing in the matrix
          const size_t e = 2 * (SP * (size_t)(it % tiles) + v % SP) + rank;
          tile_sums_out(TileSums(), red, seq++, warp - EPI_WARP0, lane,
                        partials + ((size_t)job * ptiles + e) * kNQ);
          continue;
        }
        const int r = I2 * 2 * BM + (int)rank * BM + rloc;
        const int c0 = J * BN + (int)(v % SP) * NT + half * (NT / 2);
        const int g0 = epi_first_group(r - lane, c0);
        const int curj = job == 0 ? cur0 : st->cur1[job - 1];
        const float* Sc = master + (size_t)(curj * (1 + k) + job) * mat + (size_t)c0 * Np + r;
        if (g0 < epi_groups<NT / 32>(c0, cend)) epi_load_old(olds, Sc, (int)Np, g0);
      }
      float sum[NT / 2];
#pragma unroll
      for (int i = 0; i < NT / 2; ++i) sum[i] = 0.0f;
      for (int ch = 0; ch < nchunks; ++ch) {
        const bool ok =
            mbar_wait(bar_tfull + 8 * ab.idx, ab.phase, limit_ns, abort_flag, timeout_global);
        if (!epi_all(ok && !*abort_flag)) {
          alive = false;
          break;
        }
        fence_after();
        const uint32_t ta = tmem_base + tlane + (uint32_t)(ab.idx * NT + half * (NT / 2));
        const int pc = chunk_pass(ch, cpp, passes, crev);
        const float u = pc < 2 ? u01 : cross_unscale(st, job, pc, k1);
#pragma unroll
        for (int cc = 0; cc < NT / 32; ++cc) {
          uint32_t x[16];
          tmem_ld16(ta + 16 * cc, x);
#pragma unroll
          for (int i = 0; i < 16; ++i)
            sum[16 * cc + i] = fmaf(__uint_as_float(x[i]), u, sum[16 * cc + i]);
        }
        if (ch + 1 == nchunks) break;   // keep the last chunk's buffer
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(lead_tempty + 8 * ab.idx);
        ab.next(PT::ACC);
      }
      if (!alive) break;
      // the tile's sums go back into its last chunk's buffer
      const uint32_t ta_sum = tmem_base + tlane + (uint32_t)(ab.idx * NT + half * (NT / 2));
#pragma unroll
      for (int cc = 0; cc < NT / 32; ++cc) tmem_st16(ta_sum + 16 * cc, sum + 16 * cc);
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");

      const unsigned t = it % tiles;
      int I2, J;
      pair_tile_banded(t, (int)(Np / BN), band, &I2, &J);
      const int curj = job == 0 ? cur0 : st->cur1[job - 1];
      const int e_new = job == 0 ? s0e : st->s1_exp_next[job - 1];
      const float scale_new = ldexpf(1.0f, e_new);   // exact power of two
      const float sg = (float)sigma, om = 1.0f - (float)sigma;
      const bool write = job != 0 || write0;
      const int r = I2 * 2 * BM + (int)rank * BM + rloc;
      const int c0 = J * BN + (int)(v % SP) * NT + half * (NT / 2);
      const float* Sold = master + (size_t)(curj * (1 + k) + job) * mat;
      float* Snew = master + (size_t)((curj ^ 1) * (1 + k) + job) * mat;
      const int zh_new = job == 0 ? z0n : zslice(curj ^ 1, job, 0, k);
      H16* hi_new = reinterpret_cast<H16*>(ops) + (size_t)zh_new * mat;
      H16* lo_new = reinterpret_cast<H16*>(ops) + (size_t)(zh_new + 1) * mat;

      TileSums ts;
      auto release = [&]() {   // the accumulator goes back to the MMA
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(lead_tempty + 8 * ab.idx);
      };
      rolled_tile_epilogue<CV, NT / 32, NT < BN>(ta_sum, Sold, Snew, hi_new, lo_new, lane, Np, r,
                                                 c0, cend, sg, om, scale_new, write, olds,
                                                 epi_block(red), ts, release);
      ab.next(PT::ACC);
      tile_sums_out(ts, red, seq++, warp - EPI_WARP0, lane,
                    partials + ((size_t)job * ptiles + 2 * (SP * (size_t)t + v % SP) + rank) * kNQ);
    }
  }

  // ---- teardown: both CTAs done (or aborted); free TMEM of the pair
  fence_before();
  __syncthreads();
  cluster_sync_all();
  fence_after();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                 "r"(PT::COLS));
  }
}

// ---------------------------------------------------------------------------
// Grouped pair kernel: one layer of many instances of a batch in one launch.
//
// Each instance keeps its own control block, workspace and tensor map (a
// GroupInst in device memory).  At entry every CTA reads each instance's
// plan for this layer (which jobs run) and forms the prefix sums of the
// instances' item counts (tiles x jobs) in shared memory; the items of all
// instances make one pool that the 76 CTA pairs walk round-robin, as the
// single-instance kernel walks its own items.  An item's instance is found
// by binary search over the prefix sums.  Everything an item computes --
// its tile, passes, accumulation chunks, K direction (the K-snake parity is
// taken from the round the single-instance launch would run it in) and its
// tile epilogue -- is what the single-instance kernel
// computes for it, so the results are the same bit for bit.

// largest i with first[i] <= g (first[0] = 0 <= g)
__device__ __forceinline__ int group_find(const int64_t* first, int count, int64_t g) {
  int lo = 0, hi = count - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (first[mid] <= g)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ void tensormap_acquire(const void* map) {
  asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(map) : "memory");
}

// The decoded item of a grouped launch.
struct GroupItem {
  int inst;        // instance
  int job;
  int passes;
  int kblocks;
  int cp0;         // kchunk0 of the item
  int64_t t;       // pair tile
  bool rev;        // K-snake direction
};

__device__ __forceinline__ GroupItem group_item(const GroupInst* __restrict__ inst,
                                                const int64_t* first, const uint32_t* jmask,
                                                int count, int64_t g, int k_snake, int chunk) {
  GroupItem r;
  r.inst = group_find(first, count, g);
  const GroupInst& gi = inst[r.inst];
  const int64_t loc = g - first[r.inst];
  const int64_t tiles = num_pair_tiles(gi.Np);
  r.job = job_at(jmask[r.inst], (int)(loc / tiles));
  r.t = loc % tiles;
  r.passes = job_passes(r.job, gi.k);
  r.kblocks = gi.kblocks;
  r.rev = k_snake && ((loc / gi.npairs) & 1);
  r.cp0 = kchunk0(gi.Np, r.kblocks, chunk, r.rev);
  return r;
}

// Dynamic item assignment of a grouped launch (GroupQueue): a pair takes
// its next item when its producer is ready for one, so pairs that drew short
// items take more of them.  Everything an item computes still depends on the
// item alone, so results stay bit-identical to single-instance launches.
constexpr uint32_t kNoItem = 0xFFFFFFFFu;

__device__ __forceinline__ unsigned long long claim_code(unsigned epoch, int64_t j, uint32_t g) {
  return ((unsigned long long)((epoch + 1u) & 0xFFFFFFu) << 40) |
         ((unsigned long long)((j / kQueueRing) & 0xFF) << 32) | g;
}

// Leader producer: claim the pair's j-th item and publish it.
__device__ __forceinline__ uint32_t claim_next(GroupQueue* gq, int64_t pair, int64_t j,
                                               unsigned epoch, int64_t items) {
  uint32_t g = atomicAdd(&gq->counter, 1u);
  if ((int64_t)g >= items) g = kNoItem;
  volatile unsigned long long* slot = &gq->slot[pair][j % kQueueRing];
  __threadfence();
  *slot = claim_code(epoch, j, g);
  return g;
}

// The pair's j-th item as its leader published it; false when the bounded
// wait expires (it then raises both abort flags) or another role aborted.
__device__ __forceinline__ bool claim_wait(GroupQueue* gq, int64_t pair, int64_t j,
                                           unsigned epoch, uint64_t limit_ns,
                                           volatile int* abort_smem, int* timeout_global,
                                           uint32_t* g) {
  volatile unsigned long long* slot = &gq->slot[pair][j % kQueueRing];
  const unsigned long long want = claim_code(epoch, j, 0u) >> 32;
  unsigned long long v = *slot;
  if ((v >> 32) == want) {
    *g = (uint32_t)v;
    return true;
  }
  const uint64_t t0 = gtimer();
  uint32_t it = 0;
  while (true) {
    v = *slot;
    if ((v >> 32) == want) {
      *g = (uint32_t)v;
      return true;
    }
    if ((++it & 63) == 0) {
      if (*abort_smem) return false;
      if (gtimer() - t0 > limit_ns) {
        *abort_smem = 1;
        atomicExch(timeout_global, 1);
        return false;
      }
    }
  }
}

template <bool BF16>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(NUM_THREADS, 1)
    layer_tc2_group_kernel(const GroupInst* __restrict__ inst, int count, int* group_timeout,
                           GroupQueue* gq, uint64_t limit_ns, int chunk, int k_snake, int band) {
  using CV = Cvt<BF16>;
  using PT = PairTile<BN>;
  using H16 = typename CV::T;
  extern __shared__ uint8_t smem_raw[];

  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - raw);
  const uint32_t ring = base;
  uint8_t* misc = gbase + PT::STAGES * PT::STAGE;
  int64_t* first = reinterpret_cast<int64_t*>(misc + 1024 + EPI_SCRATCH);
  uint32_t* jmask = reinterpret_cast<uint32_t*>(first + count + 1);

  const uint32_t rank = cluster_rank();
  const bool leader = rank == 0;
  const int64_t pair = blockIdx.x >> 1;

  uint64_t* bars = reinterpret_cast<uint64_t*>(misc);
  const uint32_t bar_full = smem_u32(bars);
  const uint32_t bar_empty = bar_full + 8 * PT::STAGES;
  const uint32_t bar_tfull = bar_empty + 8 * PT::STAGES;
  const uint32_t bar_tempty = bar_tfull + 8 * 2;
  const uint32_t bar_drain = bar_tempty + 8 * 2;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(misc + 256);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 264);
  float* red = reinterpret_cast<float*>(misc + 1024);
  const uint32_t lead_full = map_to_rank(bar_full, 0);
  const uint32_t lead_tempty = map_to_rank(bar_tempty, 0);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < PT::STAGES; ++s) {
      mbar_init(bar_full + 8 * s, 1);
      mbar_init(bar_empty + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar_tfull + 8 * b, 1);
      mbar_init(bar_tempty + 8 * b, 2 * EPI_WARPS);
    }
    mbar_init(bar_drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32((const void*)tmem_slot)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
  }
  fence_before();
  cluster_sync_all();   // barriers of both CTAs initialised, TMEM allocated
  fence_after();
  const uint32_t tmem_base = *tmem_slot;
  int* timeout_global = group_timeout;

  // ---- everything above ran while the decide step before finished
  pdl_wait();
  pdl_launch();
  __threadfence();   // the control blocks are read through L1

  // ---- this layer's items of every instance (same values in every CTA:
  //      the control blocks do not change during the launch)
  for (int i = threadIdx.x; i < count; i += blockDim.x) {
    const State* sti = inst[i].st;
    uint32_t jm = 0;
    if (!sti->done) {
      jm = sti->plan_square ? 1u : 0u;
      for (int j = 0; j < inst[i].k; ++j)
        if (sti->plan_resp[j]) jm |= 1u << (1 + j);
    }
    jmask[i] = jm;
    first[i + 1] = num_pair_tiles(inst[i].Np) * __popc(jm);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    first[0] = 0;
    for (int i = 0; i < count; ++i) first[i + 1] += first[i];
  }
  __syncthreads();
  const int64_t items = first[count];
  const unsigned epoch = *(volatile unsigned*)&gq->epoch;   // fixed during the launch

  if (items == 0) {
    // every instance has ended
  } else if (warp == 0) {
    // ================= TMA producer (both CTAs load their own halves) ======
    {
      RingPos rg;
      bool ok = true;
      int last_inst = -1;
      for (int64_t j = 0; ok; ++j) {
        uint32_t g = kNoItem;
        if (lane == 0) {   // kNoItem as well when the wait fails
          if (leader)
            g = claim_next(gq, pair, j, epoch, items);
          else if (!claim_wait(gq, pair, j, epoch, limit_ns, abort_flag, timeout_global, &g))
            g = kNoItem;
        }
        g = __shfl_sync(0xffffffffu, g, 0);
        if (g == kNoItem) break;
        const GroupItem itm = group_item(inst, first, jmask, count, g, k_snake, chunk);
        const GroupInst& gi = inst[itm.inst];
        if (itm.inst != last_inst) {
          tensormap_acquire(&gi.map);
          last_inst = itm.inst;
        }
        const State* sti = gi.st;
        int I2, J;
        pair_tile_banded((unsigned)itm.t, (int)(gi.Np / BN), band, &I2, &J);
        const int cols = tile_cols(J * BN, BN, itm.kblocks * BK);
        ok = produce_item<BN>(rg, &gi.map, &gi.map, sti, itm.job, itm.passes, gi.k, gi.k, sti->cur0,
                          sti->z0_cur, I2 * 2 * BM + (int)rank * BM,
                          J * BN + (int)rank * (cols / 2),
                          itm.kblocks, itm.rev, leader, ring, bar_full, bar_empty, lead_full,
                          limit_ns, abort_flag, timeout_global);
      }
      if (lane == 0) producer_drain(rg, PT::STAGES, bar_empty, limit_ns);
    }
  } else if (warp == 1) {
    // ================= MMA issuer (leader CTA only) =================
    if (leader) {
      RingPos rg, tb;
      bool ok = true;
      for (int64_t j = 0; ok; ++j) {
        uint32_t g = kNoItem;
        if (lane == 0 &&
            !claim_wait(gq, pair, j, epoch, limit_ns, abort_flag, timeout_global, &g))
          g = kNoItem;
        g = __shfl_sync(0xffffffffu, g, 0);
        if (g == kNoItem) break;
        const GroupItem itm = group_item(inst, first, jmask, count, g, k_snake, chunk);
        int I2, J;
        pair_tile_banded((unsigned)itm.t, (int)(inst[itm.inst].Np / BN), band, &I2, &J);
        ok = mma_item<BF16, BN>(rg, tb, itm.passes, itm.kblocks, chunk, itm.cp0, itm.rev,
                                tile_cols(J * BN, BN, itm.kblocks * BK),
                                tmem_base, ring, bar_full, bar_empty, bar_tfull, bar_tempty,
                                limit_ns, abort_flag, timeout_global);
      }
      if (elect_one())
        asm volatile(
            "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                bar_drain)
            : "memory");
      __syncwarp();
      const uint64_t t0 = gtimer();
      while (!mbar_try_wait(bar_drain, 0) && gtimer() - t0 < limit_ns) {
      }
    }
  } else if (warp >= EPI_WARP0) {
    // ================= epilogue (both CTAs, own 128 rows) =================
    const int q = warp & 3;
    const int half = (warp - EPI_WARP0) >> 2;
    const int rloc = 32 * q + lane;
    const uint32_t tlane = (uint32_t)(32 * q) << 16;
    int ab = 0;
    uint32_t abphase = 0;
    bool alive = true;
    uint32_t seq = 0;   // items done (tile_sums_out)
    for (int64_t j = 0; alive; ++j) {
      // lane 0 of each warp reads the claim; every epilogue warp agrees on it
      uint32_t g = kNoItem;
      bool got = true;
      if (lane == 0) got = claim_wait(gq, pair, j, epoch, limit_ns, abort_flag, timeout_global, &g);
      g = __shfl_sync(0xFFFFFFFFu, g, 0);
      got = __shfl_sync(0xFFFFFFFFu, got ? 1 : 0, 0) != 0;
      if (!epi_all(got && !*abort_flag)) {
        alive = false;
        break;
      }
      if (g == kNoItem) break;
      const GroupItem itm = group_item(inst, first, jmask, count, g, k_snake, chunk);
      const GroupInst& gi = inst[itm.inst];
      const State* sti = gi.st;
      const int job = itm.job;
      const int k = gi.k;
      const int passes = itm.passes;
      const int cpp = (itm.cp0 + itm.kblocks + chunk - 1) / chunk;   // chunks per pass
      const int nchunks = passes * cpp;
      const int s0e = sti->s0_exp;
      // exact power-of-two unscale of the products (first-order jobs and the
      // square: passes 0 and 1 only)
      const float u = ldexpf(1.0f, -(s0e + (job == 0 ? s0e : sti->s1_exp_cur[job - 1])));
      float sum[128];
#pragma unroll
      for (int i = 0; i < 128; ++i) sum[i] = 0.0f;
      for (int ch = 0; ch < nchunks; ++ch) {
        const bool ok =
            mbar_wait(bar_tfull + 8 * ab, abphase, limit_ns, abort_flag, timeout_global);
        if (!epi_all(ok && !*abort_flag)) {
          alive = false;
          break;
        }
        fence_after();
        const uint32_t ta = tmem_base + tlane + (uint32_t)(ab * BN + half * 128);
#pragma unroll
        for (int cc = 0; cc < 8; ++cc) {
          uint32_t x[16];
          tmem_ld16(ta + 16 * cc, x);
#pragma unroll
          for (int i = 0; i < 16; ++i)
            sum[16 * cc + i] = fmaf(__uint_as_float(x[i]), u, sum[16 * cc + i]);
        }
        if (ch + 1 == nchunks) break;   // keep the last chunk's buffer
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(lead_tempty + 8 * ab);
        if (++ab == 2) {
          ab = 0;
          abphase ^= 1;
        }
      }
      if (!alive) break;
      // the tile's sums go back into its last chunk's buffer (rolled epilogue)
      const uint32_t ta_sum = tmem_base + tlane + (uint32_t)(ab * BN + half * 128);
#pragma unroll
      for (int cc = 0; cc < 8; ++cc) tmem_st16(ta_sum + 16 * cc, sum + 16 * cc);
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");

      const int64_t Np = gi.Np;
      const size_t mat = (size_t)Np * Np;
      int I2, J;
      pair_tile_banded((unsigned)itm.t, (int)(Np / BN), band, &I2, &J);
      const int cur0 = sti->cur0;
      const int curj = job == 0 ? cur0 : sti->cur1[job - 1];
      const int e_new = job == 0 ? s0e : sti->s1_exp_next[job - 1];
      const float scale_new = ldexpf(1.0f, e_new);   // exact power of two
      const float sigma = (float)sti->sigma_cur;
      const float sg = sigma, om = 1.0f - sigma;
      const bool write = job != 0 || sti->plan_write0;
      const int r = I2 * 2 * BM + (int)rank * BM + rloc;
      const int c0 = J * BN + half * 128;
      float* master = gi.master;
      const float* Sold = master + (size_t)(curj * (1 + k) + job) * mat;
      float* Snew = master + (size_t)((curj ^ 1) * (1 + k) + job) * mat;
      const int zh_new = job == 0 ? sti->z0_next : zslice(curj ^ 1, job, 0, k);
      H16* hi_new = reinterpret_cast<H16*>(gi.ops) + (size_t)zh_new * mat;
      H16* lo_new = reinterpret_cast<H16*>(gi.ops) + (size_t)(zh_new + 1) * mat;

      float olds[16];
      TileSums ts;
      auto release = [&]() {   // the accumulator goes back to the MMA
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(lead_tempty + 8 * ab);
      };
      rolled_tile_epilogue<CV, 8, false>(ta_sum, Sold, Snew, hi_new, lo_new, lane, Np, r, c0,
                                         itm.kblocks * BK, sg, om, scale_new, write, olds,
                                         epi_block(red), ts, release);
      if (++ab == 2) {
        ab = 0;
        abphase ^= 1;
      }
      tile_sums_out(ts, red, seq++, warp - EPI_WARP0, lane,
                    gi.partials + ((size_t)job * gi.ptiles + 2 * itm.t + rank) * kNQ);
    }
  }

  // ---- teardown: both CTAs done (or aborted); free TMEM of the pair
  fence_before();
  __syncthreads();
  cluster_sync_all();
  fence_after();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                 "r"(TMEM_COLS));
  }
}

// ---------------------------------------------------------------------------
// Grouped pair kernel on 256 x 128 tiles (batches; option of the batch path).
//
// The same pool of items, dynamic queue and per-item work as the 256 x 256
// grouped kernel, with three changes that suit small instances:
//  - N = 128: each CTA of a pair loads 64 B rows per stage (a 64-row tensor
//    map), so a stage is 48 KB and the ring holds 4 of them (PairTile);
//  - tensor memory holds four 128-column accumulators, so a tile epilogue,
//    which keeps its tile's sums in the last chunk's accumulator while it
//    stores, leaves the MMA issuer three accumulators to run ahead with;
//  - the instances are padded to a multiple of 128 instead of 256.  A row
//    block of 256 can then extend 128 rows past the matrix: its second CTA
//    multiplies zeros (the tensor map fills rows past Np with zeros) and skips
//    its epilogue.
// Items run their K passes forwards (no K-snake): the queue keeps the items
// in flight within a few instances, whose operand panels stay in L2.  An
// instance whose 256 x 256 tiles take one round of the CTA pairs has no
// backwards sweep in the other kernels either and gets the same bits from all
// of them; larger ones agree to rounding.
constexpr int G_BN = 128;                                   // tile columns
using GT = PairTile<G_BN>;
static_assert(GT::COLS == TMEM_COLS, "accumulators fill the allocation");

// 256 x 128 tiles holding some element with row <= col: 256-row block I2 and
// 128-column block J' with J' >= 2 I2; row-major (I2, then J').
__host__ __device__ inline int64_t num_tiles128(int64_t Np) {
  const int64_t tj = Np / G_BN, t2 = (Np + 255) / 256;
  return t2 * tj - t2 * (t2 - 1);   // sum over I2 < t2 of (tj - 2 I2)
}
__device__ __forceinline__ void tile128_coords(int64_t t, int64_t Np, int* I2, int* J) {
  const int tj = (int)(Np / G_BN);
  int i = 0;
  while (t >= tj - 2 * i) {
    t -= tj - 2 * i;
    ++i;
  }
  *I2 = i;
  *J = 2 * i + (int)t;
}

struct GroupItem128 {
  int inst, job, passes, kblocks;
  int64_t t;
};

__device__ __forceinline__ GroupItem128 group_item128(const GroupInst* __restrict__ inst,
                                                      const int64_t* first, const uint32_t* jmask,
                                                      int count, int64_t g) {
  GroupItem128 r;
  r.inst = group_find(first, count, g);
  const GroupInst& gi = inst[r.inst];
  const int64_t loc = g - first[r.inst];
  const int64_t tiles = num_tiles128(gi.Np);
  r.job = job_at(jmask[r.inst], (int)(loc / tiles));
  r.t = loc % tiles;
  r.passes = job_passes(r.job, gi.k);
  r.kblocks = gi.kblocks;
  return r;
}

template <bool BF16>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(NUM_THREADS, 1)
    layer_tc2_group128_kernel(const GroupInst* __restrict__ inst, int count, int* group_timeout,
                              GroupQueue* gq, uint64_t limit_ns, int chunk) {
  using CV = Cvt<BF16>;
  using H16 = typename CV::T;
  extern __shared__ uint8_t smem_raw[];

  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - raw);
  const uint32_t ring = base;
  uint8_t* misc = gbase + GT::STAGES * GT::STAGE;
  int64_t* first = reinterpret_cast<int64_t*>(misc + 1024 + EPI_SCRATCH);
  uint32_t* jmask = reinterpret_cast<uint32_t*>(first + count + 1);

  const uint32_t rank = cluster_rank();
  const bool leader = rank == 0;
  const int64_t pair = blockIdx.x >> 1;

  uint64_t* bars = reinterpret_cast<uint64_t*>(misc);
  const uint32_t bar_full = smem_u32(bars);
  const uint32_t bar_empty = bar_full + 8 * GT::STAGES;
  const uint32_t bar_tfull = bar_empty + 8 * GT::STAGES;
  const uint32_t bar_tempty = bar_tfull + 8 * GT::ACC;
  const uint32_t bar_drain = bar_tempty + 8 * GT::ACC;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(misc + 256);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 264);
  float* red = reinterpret_cast<float*>(misc + 1024);
  const uint32_t lead_full = map_to_rank(bar_full, 0);
  const uint32_t lead_tempty = map_to_rank(bar_tempty, 0);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < GT::STAGES; ++s) {
      mbar_init(bar_full + 8 * s, 1);
      mbar_init(bar_empty + 8 * s, 1);
    }
    for (int b = 0; b < GT::ACC; ++b) {
      mbar_init(bar_tfull + 8 * b, 1);
      mbar_init(bar_tempty + 8 * b, 2 * EPI_WARPS);
    }
    mbar_init(bar_drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32((const void*)tmem_slot)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
  }
  fence_before();
  cluster_sync_all();   // barriers of both CTAs initialised, TMEM allocated
  fence_after();
  const uint32_t tmem_base = *tmem_slot;
  int* timeout_global = group_timeout;

  // ---- everything above ran while the decide step before finished
  pdl_wait();
  pdl_launch();
  __threadfence();   // the control blocks are read through L1

  // ---- this layer's items of every instance (as in the 256 x 256 kernel)
  for (int i = threadIdx.x; i < count; i += blockDim.x) {
    const State* sti = inst[i].st;
    uint32_t jm = 0;
    if (!sti->done) {
      jm = sti->plan_square ? 1u : 0u;
      for (int j = 0; j < inst[i].k; ++j)
        if (sti->plan_resp[j]) jm |= 1u << (1 + j);
    }
    jmask[i] = jm;
    first[i + 1] = num_tiles128(inst[i].Np) * __popc(jm);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    first[0] = 0;
    for (int i = 0; i < count; ++i) first[i + 1] += first[i];
  }
  __syncthreads();
  const int64_t items = first[count];
  const unsigned epoch = *(volatile unsigned*)&gq->epoch;   // fixed during the launch

  if (items == 0) {
    // every instance has ended
  } else if (warp == 0) {
    // ================= TMA producer (both CTAs load their own rows) ======
    {
      RingPos rg;
      bool ok = true;
      int last_inst = -1;
      for (int64_t j = 0; ok; ++j) {
        uint32_t g = kNoItem;
        if (lane == 0) {   // kNoItem as well when the wait fails
          if (leader)
            g = claim_next(gq, pair, j, epoch, items);
          else if (!claim_wait(gq, pair, j, epoch, limit_ns, abort_flag, timeout_global, &g))
            g = kNoItem;
        }
        g = __shfl_sync(0xffffffffu, g, 0);
        if (g == kNoItem) break;
        const GroupItem128 itm = group_item128(inst, first, jmask, count, g);
        const GroupInst& gi = inst[itm.inst];
        if (itm.inst != last_inst) {
          tensormap_acquire(&gi.map);
          tensormap_acquire(&gi.map64);
          last_inst = itm.inst;
        }
        const State* sti = gi.st;
        int I2, J;
        tile128_coords(itm.t, gi.Np, &I2, &J);
        const int cols = tile_cols(J * G_BN, G_BN, itm.kblocks * BK);
        ok = produce_item<G_BN>(rg, &gi.map, &gi.map64, sti, itm.job, itm.passes, gi.k, gi.k,
                                sti->cur0, sti->z0_cur, I2 * 2 * BM + (int)rank * BM,
                                J * G_BN + (int)rank * (cols / 2), itm.kblocks, false, leader,
                                ring, bar_full, bar_empty, lead_full, limit_ns, abort_flag,
                                timeout_global);
      }
      if (lane == 0) producer_drain(rg, GT::STAGES, bar_empty, limit_ns);
    }
  } else if (warp == 1) {
    // ================= MMA issuer (leader CTA only) =================
    if (leader) {
      RingPos rg, tb;
      bool ok = true;
      for (int64_t j = 0; ok; ++j) {
        uint32_t g = kNoItem;
        if (lane == 0 &&
            !claim_wait(gq, pair, j, epoch, limit_ns, abort_flag, timeout_global, &g))
          g = kNoItem;
        g = __shfl_sync(0xffffffffu, g, 0);
        if (g == kNoItem) break;
        const GroupItem128 itm = group_item128(inst, first, jmask, count, g);
        int I2, J;
        tile128_coords(itm.t, inst[itm.inst].Np, &I2, &J);
        ok = mma_item<BF16, G_BN>(rg, tb, itm.passes, itm.kblocks, chunk, 0, false,
                                  tile_cols(J * G_BN, G_BN, itm.kblocks * BK),
                                  tmem_base, ring, bar_full, bar_empty, bar_tfull, bar_tempty,
                                  limit_ns, abort_flag, timeout_global);
      }
      if (elect_one())
        asm volatile(
            "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                bar_drain)
            : "memory");
      __syncwarp();
      const uint64_t t0 = gtimer();
      while (!mbar_try_wait(bar_drain, 0) && gtimer() - t0 < limit_ns) {
      }
    }
  } else if (warp >= EPI_WARP0) {
    // ========== epilogue (both CTAs, own 128 rows; warps split 64 + 64 columns) ==========
    const int q = warp & 3;
    const int half = (warp - EPI_WARP0) >> 2;
    const int rloc = 32 * q + lane;
    const uint32_t tlane = (uint32_t)(32 * q) << 16;
    RingPos ab;
    bool alive = true;
    uint32_t seq = 0;   // items done (tile_sums_out)
    for (int64_t j = 0; alive; ++j) {
      uint32_t g = kNoItem;
      bool got = true;
      if (lane == 0) got = claim_wait(gq, pair, j, epoch, limit_ns, abort_flag, timeout_global, &g);
      g = __shfl_sync(0xFFFFFFFFu, g, 0);
      got = __shfl_sync(0xFFFFFFFFu, got ? 1 : 0, 0) != 0;
      if (!epi_all(got && !*abort_flag)) {
        alive = false;
        break;
      }
      if (g == kNoItem) break;
      const GroupItem128 itm = group_item128(inst, first, jmask, count, g);
      const GroupInst& gi = inst[itm.inst];
      const State* sti = gi.st;
      const int job = itm.job;
      const int k = gi.k;
      const int cpp = (itm.kblocks + chunk - 1) / chunk;   // chunks per pass
      const int nchunks = itm.passes * cpp;
      const int s0e = sti->s0_exp;
      // exact power-of-two unscale of the products (first-order jobs and the
      // square: passes 0 and 1 only)
      const float u = ldexpf(1.0f, -(s0e + (job == 0 ? s0e : sti->s1_exp_cur[job - 1])));
      float sum[64];
#pragma unroll
      for (int i = 0; i < 64; ++i) sum[i] = 0.0f;
      for (int ch = 0; ch < nchunks; ++ch) {
        const bool ok =
            mbar_wait(bar_tfull + 8 * ab.idx, ab.phase, limit_ns, abort_flag, timeout_global);
        if (!epi_all(ok && !*abort_flag)) {
          alive = false;
          break;
        }
        fence_after();
        const uint32_t ta = tmem_base + tlane + (uint32_t)(ab.idx * G_BN + half * 64);
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
          uint32_t x[16];
          tmem_ld16(ta + 16 * cc, x);
#pragma unroll
          for (int i = 0; i < 16; ++i)
            sum[16 * cc + i] = fmaf(__uint_as_float(x[i]), u, sum[16 * cc + i]);
        }
        if (ch + 1 == nchunks) break;   // keep the last chunk's accumulator
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(lead_tempty + 8 * ab.idx);
        ab.next(GT::ACC);
      }
      if (!alive) break;
      // the tile's sums go back into its last chunk's accumulator (rolled epilogue)
      const uint32_t ta_sum = tmem_base + tlane + (uint32_t)(ab.idx * G_BN + half * 64);
#pragma unroll
      for (int cc = 0; cc < 4; ++cc) tmem_st16(ta_sum + 16 * cc, sum + 16 * cc);
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");

      const int64_t Np = gi.Np;
      const size_t mat = (size_t)Np * Np;
      int I2, J;
      tile128_coords(itm.t, Np, &I2, &J);
      const int cur0 = sti->cur0;
      const int curj = job == 0 ? cur0 : sti->cur1[job - 1];
      const int e_new = job == 0 ? s0e : sti->s1_exp_next[job - 1];
      const float scale_new = ldexpf(1.0f, e_new);   // exact power of two
      const float sigma = (float)sti->sigma_cur;
      const float sg = sigma, om = 1.0f - sigma;
      const bool write = job != 0 || sti->plan_write0;
      const int row0 = I2 * 2 * BM + (int)rank * BM;   // this CTA's first row
      const int r = row0 + rloc;
      const int c0 = J * G_BN + half * 64;
      float* master = gi.master;
      const float* Sold = master + (size_t)(curj * (1 + k) + job) * mat;
      float* Snew = master + (size_t)((curj ^ 1) * (1 + k) + job) * mat;
      const int zh_new = job == 0 ? sti->z0_next : zslice(curj ^ 1, job, 0, k);
      H16* hi_new = reinterpret_cast<H16*>(gi.ops) + (size_t)zh_new * mat;
      H16* lo_new = reinterpret_cast<H16*>(gi.ops) + (size_t)(zh_new + 1) * mat;

      float olds[16];
      TileSums ts;
      auto release = [&]() {   // the accumulator goes back to the MMA
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(lead_tempty + 8 * ab.idx);
      };
      // rows past Np (a 256-row block over a matrix padded to 128): nothing to
      // store; the products there are zeros
      if ((int64_t)row0 < Np)
        rolled_tile_epilogue<CV, 4, false>(ta_sum, Sold, Snew, hi_new, lo_new, lane, Np, r, c0,
                                           itm.kblocks * BK, sg, om, scale_new, write, olds,
                                           epi_block(red), ts, release);
      else
        release();
      ab.next(GT::ACC);
      tile_sums_out(ts, red, seq++, warp - EPI_WARP0, lane,
                    gi.partials + ((size_t)job * gi.ptiles + 2 * itm.t + rank) * kNQ);
    }
  }

  // ---- teardown: both CTAs done (or aborted); free TMEM of the pair
  fence_before();
  __syncthreads();
  cluster_sync_all();
  fence_after();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                 "r"(TMEM_COLS));
  }
}

// ---------------------------------------------------------------------------
// Host side

using PairKernel = decltype(&layer_tc2_kernel<false, BN>);
PairKernel pair_kernel(bool bf16, int nt) {
  if (nt == 64) return bf16 ? layer_tc2_kernel<true, 64> : layer_tc2_kernel<false, 64>;
  if (nt == 128) return bf16 ? layer_tc2_kernel<true, 128> : layer_tc2_kernel<false, 128>;
  return bf16 ? layer_tc2_kernel<true, BN> : layer_tc2_kernel<false, BN>;
}

int pair_smem(int nt) {
  return nt == 64 ? PairTile<64>::SMEM : (nt == 128 ? PairTile<128>::SMEM : PairTile<BN>::SMEM);
}

// Tile width of the pair kernel for `tiles` 256 x 256 tiles of each job.
// Measured time per layer in us of a whole solve, 256 / 128 / 64 wide:
//   n = 128 k = 1   29 /  22 /  20       n = 2048 k = 1   84 /  74 / 106
//   n = 768 k = 1   45 /  31 /  29       n = 2048 k = 3  155 / 150 / 224
//   n = 768 k = 3   46 /  33 /  37       n = 2560 k = 3  270 / 285 / 397
//   n = 1280 k = 3  64 /  66 /  86       n = 3072 k = 1  256 / 228 / 314
// 64: while one round of the pairs holds every tile; the tile's own time (its
// epilogue above all) is then what counts.  Above, the busiest pair's load
// decides: a 128-wide tile takes 0.6 of the time of a 256-wide one per K block
// (it loads 24 KB per 32-wide block for half the products, and its MMAs issue
// no faster than 0.24 us per block against 0.4), and its last epilogue is
// about 14 blocks shorter.  The pairs take the items round-robin, responses
// (two K passes; those of higher orders, which have more, are counted alike)
// first, so pair 0 has the largest load.
// The jobs are those that run, not the layout's slots: a density forward runs
// the square alone, its backward one response, a replay the responses alone
// (whole calls in ms, by the width for the slots and a square / by the jobs:
// forward with a checkpoint every eight states n = 1280 1.09 / 1.02, 2560 2.52 /
// 2.43, 3584 5.30 / 4.79; its backward 1.99 / 1.87, 5.51 / 5.28, 12.5 / 11.0;
// replay n = 1536 k = 3 2.71 / 2.59, 2304 k = 1 3.58 / 3.38).
int pair_tile_width(int64_t tiles, const LayerJobs& jobs, int64_t kblocks, int pairs) {
  const int64_t items = tiles * (jobs.responses + (jobs.square ? 1 : 0));
  if (BN / 64 * items <= pairs) return 64;
  if (items > 8 * pairs) return BN;
  auto load = [&](int split) {
    int64_t passes = 0;
    for (int64_t i = 0; i < split * items; i += pairs)
      passes += i < split * tiles * jobs.responses ? 2 : 1;
    return passes * kblocks;
  };
  return 3 * load(2) < 5 * (load(1) + 14) ? 128 : BN;
}

// Per-device one-time setup of the tensor-core kernels (their shared-memory
// attribute is set in each device's context) and the device's SM count;
// thread-safe.
constexpr int kMaxDevices = 64;
struct DeviceSetup {
  std::once_flag once;
  int sms = 0;
};
int device_setup() {
  static DeviceSetup tab[kMaxDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 0;
  DeviceSetup& d = tab[dev];
  std::call_once(d.once, [&] {
    cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, dev);
    cudaFuncSetAttribute(layer_tc_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         SMEM_BYTES);
    cudaFuncSetAttribute(layer_tc_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         SMEM_BYTES);
    for (bool bf16 : {false, true})
      for (int nt : {256, 128, 64})
        cudaFuncSetAttribute(pair_kernel(bf16, nt), cudaFuncAttributeMaxDynamicSharedMemorySize,
                             pair_smem(nt));
    constexpr int ring_smem =
        PairTile<BN>::SMEM > GT::SMEM ? PairTile<BN>::SMEM : GT::SMEM;
    constexpr int group_smem = ring_smem + (kGroupMax + 1) * (int)sizeof(int64_t) +
                               kGroupMax * (int)sizeof(uint32_t);
    static_assert(group_smem <= 227 * 1024, "grouped kernel shared memory");
    cudaFuncSetAttribute(layer_tc2_group_kernel<false>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, group_smem);
    cudaFuncSetAttribute(layer_tc2_group_kernel<true>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, group_smem);
    cudaFuncSetAttribute(layer_tc2_group128_kernel<false>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, group_smem);
    cudaFuncSetAttribute(layer_tc2_group128_kernel<true>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, group_smem);
  });
  return d.sms;
}

PFN_cuTensorMapEncodeTiled_v12000 get_encoder() {
  // looked up once per process (thread-safe static initialisation)
  static const PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    return (PFN_cuTensorMapEncodeTiled_v12000) nullptr;
  }();
  return fn;
}

// sk: K elements per box (32 or 64: 64- or 128-byte swizzle)
bool make_map(CUtensorMap* map, void* base, int64_t Np, int slices, int box_rows, bool bf16,
              int sk) {
  auto enc = get_encoder();
  if (!enc) return false;
  cuuint64_t dims[3] = {(cuuint64_t)Np, (cuuint64_t)Np, (cuuint64_t)slices};
  cuuint64_t strides[2] = {(cuuint64_t)Np * 2, (cuuint64_t)Np * Np * 2};
  cuuint32_t box[3] = {(cuuint32_t)sk, (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(map, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16,
                   3, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   sk == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

}  // namespace tc

void pair_tile_info(const Layout& L, int64_t* entries, double* pass_flops, bool n128) {
  const int64_t tiles = n128 ? tc::num_tiles128(L.Np) : tc::num_pair_tiles(L.Np);
  // the last column block's tiles are as wide as what is left of the matrix
  const int nt = n128 ? tc::G_BN : tc::BN;
  const int64_t edge = n128 ? (L.Np + 255) / 256 : L.Np / tc::BN;
  const int cend = tc::k_blocks(L.n) * tc::BK;
  const double cols = nt - (double)edge / tiles * (L.Np - cend);
  if (entries) *entries = 2 * tiles;
  if (pass_flops)
    *pass_flops = (double)tiles * 2 * tc::BM * cols * tc::k_blocks(L.n) * tc::BK * 2.0;
}

bool make_group_inst(const Layout& L, void* ws, int sm_count, GroupInst* gi, bool n128) {
  using namespace tc;
  char* base = (char*)ws;
  const bool bf16 = L.precision == DMPT_DUAL_BF16;
  const int slices = 2 * (1 + L.k) * 2 + 2 * L.tape_states;
  if (!make_map(&gi->map, base + L.off_ops16, L.Np, slices, BM, bf16, GT::SK)) return false;
  if (n128 && !make_map(&gi->map64, base + L.off_ops16, L.Np, slices, GT::B_ROWS, bf16, GT::SK))
    return false;
  gi->st = (State*)(base + L.off_state);
  gi->master = (float*)(base + L.off_master);
  gi->ops = (uint16_t*)(base + L.off_ops16);
  gi->partials = (double*)(base + L.off_partials);
  gi->Np = L.Np;
  gi->kblocks = k_blocks(L.n);
  gi->ptiles = L.partial_tiles;
  gi->k = L.k;
  const int64_t max_items = num_pair_tiles(L.Np) * (1 + L.k);
  int64_t pairs = sm_count / 2;
  if (pairs > max_items) pairs = max_items;
  gi->npairs = (int)pairs;
  return true;
}

cudaError_t launch_layer_tc_group(const GroupInst* inst, int count, bool bf16, int* group_timeout,
                                  GroupQueue* queue, double timeout_s, int accum_chunk_k,
                                  int k_snake, int band, int sm_count, cudaStream_t s,
                                  bool n128) {
  using namespace tc;
  if (count < 1 || count > kGroupMax || !queue || sm_count / 2 > kQueuePairs)
    return cudaErrorInvalidValue;
  const int smem = (n128 ? GT::SMEM : PairTile<BN>::SMEM) + (count + 1) * (int)sizeof(int64_t) +
                   count * (int)sizeof(uint32_t);
  if (device_setup() == 0) return cudaErrorInvalidDevice;
  const uint64_t limit_ns = (uint64_t)(timeout_s * 1e9);
  const int ck = accum_chunk_k > 0 ? accum_chunk_k : DEFAULT_CHUNK_K;
  const int chunk = ck / BK < 1 ? 1 : ck / BK;
  const int grid = 2 * (sm_count / 2);
  if (n128)
    return launch_pdl(bf16 ? layer_tc2_group128_kernel<true> : layer_tc2_group128_kernel<false>,
                      dim3(grid), dim3(NUM_THREADS), smem, s, inst, count, group_timeout, queue,
                      limit_ns, chunk);
  return launch_pdl(bf16 ? layer_tc2_group_kernel<true> : layer_tc2_group_kernel<false>,
                    dim3(grid), dim3(NUM_THREADS), smem, s, inst, count, group_timeout, queue,
                    limit_ns, chunk, k_snake, band);
}

cudaError_t launch_layer_tc(const Layout& L, void* ws, cudaStream_t s, double timeout_s,
                            int accum_chunk_k, int cta_pair, int k_snake, int band,
                            const LayerJobs& jobs, int64_t* entries, double* pass_flops,
                            int inject_stall, int round_align) {
  using namespace tc;
  char* base = (char*)ws;
  const bool bf16 = L.precision == DMPT_DUAL_BF16;
  const int slices = 2 * (1 + L.k) * 2 + 2 * L.tape_states;
  CUtensorMap mA, mB;
  const int sms = device_setup();
  if (sms == 0) return cudaErrorInvalidDevice;
  // 256 x 256 tiles of every slot; `jobs` of them run at first (which ones still
  // do is only known on the device)
  const int64_t ptiles = num_pair_tiles(L.Np), pitems = ptiles * (1 + L.k);
  const int nt = pair_tile_width(ptiles, jobs, k_blocks(L.n), sms / 2);
  const int sk = cta_pair ? PairTile<BN>::SK : BK;
  if (!make_map(&mA, base + L.off_ops16, L.Np, slices, BM, bf16, sk) ||
      !make_map(&mB, base + L.off_ops16, L.Np, slices, cta_pair ? nt / 2 : BN, bf16, sk))
    return cudaErrorInvalidValue;
  const uint64_t limit_ns = (uint64_t)(timeout_s * 1e9);
  int ck = accum_chunk_k > 0 ? accum_chunk_k : DEFAULT_CHUNK_K;
  int chunk = ck / BK;
  if (chunk < 1) chunk = 1;
  State* st = (State*)(base + L.off_state);
  float* master = (float*)(base + L.off_master);
  uint16_t* ops = (uint16_t*)(base + L.off_ops16);
  double* partials = (double*)(base + L.off_partials);
  if (cta_pair) {
    const int split = BN / nt;
    const int64_t max_items = split * pitems;
    const int pairs = (int)(max_items < sms / 2 ? max_items : sms / 2);
    const int snake_pairs = (int)(pitems < sms / 2 ? pitems : sms / 2);
    const cudaError_t e = launch_pdl(
        pair_kernel(bf16, nt), dim3(2 * pairs), dim3(NUM_THREADS), pair_smem(nt), s, mA, mB, st,
        master, ops, L.Np, L.k, partials, L.partial_tiles, limit_ns, chunk, k_snake, snake_pairs,
        band, inject_stall, round_align);
    if (e != cudaSuccess) return e;
    if (entries) *entries = 2 * split * ptiles;
    pair_tile_info(L, nullptr, pass_flops);
    return cudaGetLastError();
  }
  const int64_t tiles = num_tiles(L.Np);
  // the number of jobs is only known on the device; size the grid for the
  // largest case and let surplus CTAs exit
  int64_t max_items = tiles * (1 + L.k);
  int grid = (int)(max_items < sms ? max_items : sms);
  if (bf16)
    layer_tc_kernel<true><<<grid, NUM_THREADS, SMEM_BYTES, s>>>(mA, mB, st, master, ops, L.Np,
                                                                L.k, partials, L.partial_tiles,
                                                                limit_ns, chunk, inject_stall);
  else
    layer_tc_kernel<false><<<grid, NUM_THREADS, SMEM_BYTES, s>>>(mA, mB, st, master, ops, L.Np,
                                                                 L.k, partials, L.partial_tiles,
                                                                 limit_ns, chunk, inject_stall);
  if (entries) *entries = tiles;
  if (pass_flops) *pass_flops = (double)tiles * BM * BN * k_blocks(L.n) * BK * 2.0;
  return cudaGetLastError();
}

}  // namespace dmpt

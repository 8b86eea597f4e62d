// Element-wise kernels, device-side control of Algorithms 1-3, and the SIMT
// (FP64 / FP32) layer product with its fused epilogue.
//
// Matrices inside the workspace are n x n in a stride of Np, the multiple of 256
// (128 on the 256 x 128 tiles of a batch) at or above n.  The initial kernels
// write all Np x Np elements, zeros outside the matrix; zeros are invariant
// under the SP2 layers (0^2 = 0, 2*0 - 0^2 = 0) and add nothing to traces or
// norms.  The layer products work on the blocks that hold rows and columns < n
// (the FP64 form on those elements alone), so what lies beyond is not kept up.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <math.h>
#include <stddef.h>

#include <mutex>

#include "dmpt_internal.cuh"

namespace dmpt {

static inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

Layout make_layout(int64_t n, int k, int precision, int tape_states, int ckpt_slots, int pad) {
  Layout L{};
  L.n = n;
  L.Np = ((n + pad - 1) / pad) * pad;
  L.k = k;
  L.precision = precision;
  L.tape_states = tape_states;
  L.elem = (precision == DMPT_FP64) ? 8 : 4;
  size_t off = 0;
  L.off_state = off;
  off = align256(off + sizeof(State));
  // one partial entry per upper tile of the smallest product tile (64; the
  // FP64 form's own) or per block of the init kernel, whichever is larger
  const int64_t tiles = precision == DMPT_FP64 ? fp64_tiles(n) : upper_tiles(L.Np, 64);
  L.partial_tiles = tiles > kInitBlocks ? tiles : kInitBlocks;
  L.off_partials = off;
  off = align256(off + (size_t)(1 + k) * (size_t)L.partial_tiles * kNQ * sizeof(double));
  const size_t mat = (size_t)L.Np * (size_t)L.Np;
  L.off_master = off;
  off = align256(off + 2 * (size_t)(1 + k) * mat * L.elem);
  if (precision == DMPT_DUAL_FP16 || precision == DMPT_DUAL_BF16) {
    L.off_ops16 = off;
    off = align256(off + (2 * (size_t)(1 + k) * 2 + 2 * (size_t)tape_states) * mat * 2);
  } else {
    L.off_ops16 = 0;
  }
  // small vectors of the self-consistent response: q[k][n], v[k][n], red[k][4]
  L.off_vec = off;
  off = align256(off + ((size_t)(k > 0 ? k : 1) * (2 * (size_t)n + 4)) * sizeof(double));
  // FP32 checkpoints of every ckpt_k-th S0 state (adjoint with recompute)
  L.ckpt_slots = ckpt_slots;
  L.off_ckpt = off;
  off = align256(off + (size_t)ckpt_slots * mat * 4);
  L.total = off;
  return L;
}

// ---------------------------------------------------------------------------
// Deterministic block reduction of NV doubles (fixed tree, fixed order).
template <int NV, int NT>
__device__ __forceinline__ void block_sum(double (&v)[NV], double* smem /* NT*NV */) {
  const int tid = threadIdx.x;
#pragma unroll
  for (int i = 0; i < NV; ++i) smem[i * NT + tid] = v[i];
  __syncthreads();
  for (int s = NT / 2; s > 0; s >>= 1) {
    if (tid < s) {
#pragma unroll
      for (int i = 0; i < NV; ++i) smem[i * NT + tid] += smem[i * NT + tid + s];
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < NV; ++i) v[i] = smem[i * NT];
  __syncthreads();
}

// ---------------------------------------------------------------------------
// Conversions between FP32 and FP64 on the integer pipe.  The part converts two
// values per clock and SM on its FP64 pipe, which bounded the initial layer (68%
// of that pipe's peak at n = 4096, 41% of DRAM's) and the outputs; these take
// about ten integer instructions (outputs n = 5904 k = 1: 503 -> 146 us, initial
// layer n = 2048 k = 3: 62 -> 46 us).  Subnormal, infinite and NaN values, and
// results outside the normal FP32 range, take the conversion instruction.

__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x), a = u & 0x7FFFFFFFu;
  if (a - 0x00800000u < 0x7F000000u)   // normal: rebias the exponent by 1023 - 127
    return __hiloint2double((int)((u & 0x80000000u) | ((a >> 3) + 0x38000000u)), (int)(u << 29));
  return a == 0u ? __hiloint2double((int)u, 0) : (double)x;
}

// (float)(x 2^-HALF), rounded to nearest even
template <int HALF = 0>
__device__ __forceinline__ float narrow(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned a = hi & 0x7FFFFFFFu;
  constexpr unsigned kOne = 0x00100000u;   // one in the exponent
  if (a - (0x38100000u + HALF * kOne) < 0x0FE00000u) {
    unsigned m = __funnelshift_l(lo, a - (0x38000000u + HALF * kOne), 3);
    m += (lo & 0x1FFFFFFFu) + (m & 1u) > 0x10000000u ? 1u : 0u;   // may carry into infinity
    return __uint_as_float((hi & 0x80000000u) | m);
  }
  return (a | lo) == 0u ? __uint_as_float(hi) : (float)(HALF ? 0.5 * x : x);
}

// ---------------------------------------------------------------------------
// Gershgorin bounds (Sec. II B; Alg. 1 inputs).  Min / max are taken with
// 64-bit integer atomics on an order-preserving encoding of the doubles, so
// the result is independent of the order in which rows finish and the call
// needs no scratch memory beyond its 2-double output.

__device__ __forceinline__ long long dkey(double x) {
  long long b = __double_as_longlong(x);
  return b >= 0 ? b : (b ^ 0x7FFFFFFFFFFFFFFFLL);
}
__device__ __forceinline__ double dkey_inv(long long k) {
  long long b = k >= 0 ? k : (k ^ 0x7FFFFFFFFFFFFFFFLL);
  return __longlong_as_double(b);
}

__global__ void bounds_init_kernel(long long* key) {
  key[0] = dkey(INFINITY);
  key[1] = dkey(-INFINITY);
}

// one warp per row; row r: centre H_rr, radius sum_{j != r} |H_rj|.  With a
// counter (zero on entry and on return) the last block to finish turns the
// keys into the bounds.
__global__ void bounds_rows_kernel(const double* __restrict__ H, int64_t n, int64_t ld,
                                   long long* key, unsigned* counter) {
  pdl_wait();
  pdl_launch();
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  double lo = INFINITY, hi = -INFINITY;
  for (int64_t r = warp; r < n; r += nwarps) {
    const double* row = H + r * ld;
    double s = 0.0;
    for (int64_t j = lane; j < n; j += 32) s += fabs(row[j]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const double d = row[r];
    const double rad = s - fabs(d);
    lo = fmin(lo, d - rad);
    hi = fmax(hi, d + rad);
  }
  if (lane == 0 && warp < n) {
    atomicMin(&key[0], dkey(lo));
    atomicMax(&key[1], dkey(hi));
  }
  if (counter == nullptr) return;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(counter, 1u) == gridDim.x - 1) {
      __threadfence();
      double* out = reinterpret_cast<double*>(key);
      const double b0 = dkey_inv(__ldcg(&key[0])), b1 = dkey_inv(__ldcg(&key[1]));
      out[0] = b0;
      out[1] = b1;
      *counter = 0u;
    }
  }
}

__global__ void bounds_fin_kernel(long long* key) {
  double lo = dkey_inv(key[0]);
  double hi = dkey_inv(key[1]);
  double* out = reinterpret_cast<double*>(key);
  out[0] = lo;
  out[1] = hi;
}

static int bounds_blocks(int64_t n) {
  const int64_t warps = n < 152 * 64 ? n : 152 * 64;
  return (int)((warps * 32 + 255) / 256);
}

cudaError_t launch_bounds(const double* H, int64_t n, int64_t ld, double* eps_out,
                          cudaStream_t s) {
  long long* key = reinterpret_cast<long long*>(eps_out);
  bounds_init_kernel<<<1, 1, 0, s>>>(key);
  bounds_rows_kernel<<<bounds_blocks(n), 256, 0, s>>>(H, n, ld, key, nullptr);
  bounds_fin_kernel<<<1, 1, 0, s>>>(key);
  return cudaGetLastError();
}

// A fresh control block of a forward run (zeroed, then its fields) with the
// keys of the bounds.
__global__ void __launch_bounds__(256)
    forward_setup_kernel(State* st, int k, int max_layers, int precision, double n_occ,
                         double c_pt, double c_d0, int tape, int tape_base, int tape_states,
                         int layout_k, int64_t n, int order, int k1, FwdOpts fo, int hole) {
  static_assert(sizeof(State) % 4 == 0, "State zeroed as words");
  pdl_launch();
  unsigned* w = reinterpret_cast<unsigned*>(st);
  for (int i = threadIdx.x; i < (int)(sizeof(State) / 4); i += blockDim.x) w[i] = 0u;
  __syncthreads();
  if (threadIdx.x == 0) {
    state_init_fields(st, k, max_layers, precision, n_occ, c_pt, c_d0, tape, tape_base,
                      tape_states, layout_k, n, order, k1, fo, hole);
    long long* key = reinterpret_cast<long long*>(&st->eps1);
    key[0] = dkey(INFINITY);
    key[1] = dkey(-INFINITY);
  }
}

cudaError_t launch_forward_setup(const Layout& L, void* ws, const double* H, int64_t ld, int slots,
                                 int max_layers, double n_occ, double c_pt, double c_d0, int tape,
                                 int order, int k1, FwdOpts fo, int hole, cudaStream_t s) {
  State* st = (State*)((char*)ws + L.off_state);
  forward_setup_kernel<<<1, 256, 0, s>>>(st, slots, max_layers, L.precision, n_occ, c_pt, c_d0,
                                         tape, 4 * (1 + L.k), L.tape_states, L.k, L.n, order, k1,
                                         fo, hole);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_pdl(bounds_rows_kernel, dim3(bounds_blocks(L.n)), dim3(256), 0, s, H, L.n, ld,
                    reinterpret_cast<long long*>(&st->eps1), &st->round_ctr);
}

// ---------------------------------------------------------------------------
// Initial normalisation layer (Alg. 1; Sec. III A, S_0(lambda)):
//   S0 = (eps_N I - H) / (eps_N - eps_1),  S1_k = -H1_k / (eps_N - eps_1).
// Only the upper triangle (j >= i) of H and H1 is read, so the stored
// matrices are exactly symmetric.  Partial sums per block: Tr S0, ||S0||_F^2,
// ||S1_k||_F^2 and a count of non-finite values.

// Block vb of vgrid blocks (256 threads): tile pairs vb, vb + vgrid, ... of
// matrices m_lo .. m_hi in turn (0 = S0, m = S1_m; those above k are the
// higher-order slots, which start at zero: a linear perturbation has H^(o) = 0
// for o >= 2).  The count of non-finite values goes with job m_lo.
template <typename T>
__device__ __forceinline__ void init_body(State* st, T* master, const double* __restrict__ H,
                                          const double* __restrict__ H1, int64_t n, int64_t Np,
                                          int64_t ld, int k, int m_lo, int m_hi,
                                          const double* __restrict__ shift, double* partials,
                                          int64_t ptiles, int64_t vb, int64_t vgrid) {
  // 64 x 64 tile pairs (bi <= bj): the upper tile is read row-wise (coalesced,
  // every load of the tile in flight at once), written in place and, through
  // shared memory, transposed into the mirror tile, so both triangles of S
  // come from the upper triangle of the input.  Each value is formed in FP64
  // and rounded once to T (for T = float, the off-diagonal values are formed
  // in FP32).  The squared norms are summed in FP64 for the FP64 form; for
  // T = float, as exact FP32 products with TwoSum compensation (the FP64 rate
  // of the part is low).
  constexpr bool F32 = sizeof(T) == 4;
  constexpr int TS = kInitTile;
  constexpr int RPT = TS * TS / 256;   // rows of the tile per thread
  constexpr int RS = TS / RPT;         // row step between them
  __shared__ T tile[TS][TS + 1];
  __shared__ double red[2 * 256];
  const double e1 = st->eps1, eN = st->epsN;
  __shared__ double w_sh;   // one FP64 division per block
  if (threadIdx.x == 0) w_sh = 1.0 / (eN - e1);
  __syncthreads();
  const double w = w_sh;
  const float wf = (float)w;
  const bool hole = st->hole != 0;   // complement form: S_0 = I - (eps_N I - H) w
  const size_t mat = (size_t)Np * Np;
  const int tx = threadIdx.x % TS, ty = threadIdx.x / TS;   // 64 x 4 threads
  const int64_t TB = Np / TS;
  const int64_t pairs = TB * (TB + 1) / 2;
  int nbad = 0;
  for (int m = m_lo; m <= m_hi && m <= k; ++m) {
    const double* src = m == 0 ? H : H1 + (size_t)(m - 1) * n * ld;
    T* dst = master + (size_t)m * mat;   // buffer 0 (slots 0 .. layout k)
    double tr = 0.0, fd = 0.0;
    float fs = 0.0f, fc = 0.0f;
    for (int64_t tp = vb; tp < pairs; tp += vgrid) {
      // tile pair index -> (bi, bj), bj-major: tp = bj (bj + 1) / 2 + bi (an
      // FP32 estimate of bj, corrected in integers)
      int64_t bj = (int64_t)((sqrtf(8.0f * (float)tp + 1.0f) - 1.0f) * 0.5f);
      while ((bj + 1) * (bj + 2) / 2 <= tp) ++bj;
      while (bj * (bj + 1) / 2 > tp) --bj;
      const int64_t bi = tp - bj * (bj + 1) / 2;
      double hv[RPT];
      {
        const int64_t r0 = bi * TS + ty, c = bj * TS + tx;
        const double* sp = src + r0 * ld + c;
        // row r0 + RS i lies in the matrix when RS i < lim
        const int lim = c < n ? (int)min((int64_t)TS, n - r0) : 0;
#pragma unroll
        for (int i = 0; i < RPT; ++i) hv[i] = RS * i < lim ? sp[(int64_t)(RS * i) * ld] : 0.0;
      }
      if constexpr (F32) {
        // off the diagonal in FP32 arithmetic (the FP64 rate of the part is
        // low): v = -+ fl32(h) w32, within 1.5 units in the last place; zero
        // outside the matrix (h = 0 there)
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
          const float hw = narrow(hv[i]) * wf;
          tile[ty + RS * i][tx] = hole ? hw : -hw;
        }
        // the diagonal element of column tx, formed in FP64 and rounded once
        if (bi == bj && tx % RS == ty) {
          const int64_t r = bi * TS + tx;
          if (r < n) {
            double h = src[r * ld + r];
            if (m > 0 && shift != nullptr) h += shift[(size_t)(m - 1) * n + r];
            const double x = hole ? (m == 0 ? (h - e1) * w : h * w)
                                  : (m == 0 ? (eN - h) * w : -h * w);
            const float xv = (float)x;
            tile[tx][tx] = xv;
            if (m == 0) tr += (double)xv;
          }
        }
      } else {
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
          const int rl = ty + RS * i;
          const int64_t r = bi * TS + rl, c = bj * TS + tx;
          double x = 0.0;
          if (r < n && c < n) {
            double h = hv[i];
            if (m > 0 && shift != nullptr && r == c) h += shift[(size_t)(m - 1) * n + r];
            if (hole)
              x = m == 0 ? (h - (r == c ? e1 : 0.0)) * w : h * w;
            else
              x = m == 0 ? ((r == c ? eN : 0.0) - h) * w : -h * w;
          }
          tile[rl][tx] = (T)x;
          if (m == 0 && r == c) tr += x;
        }
      }
      __syncthreads();
#pragma unroll 4
      for (int i = 0; i < RPT; ++i) {
        const int rl = ty + RS * i;
        const int64_t r = bi * TS + rl, c = bj * TS + tx;
        // diagonal tile: the lower half mirrors the upper half
        const T v = (bi < bj || rl <= tx) ? tile[rl][tx] : tile[tx][rl];
        dst[(size_t)r * Np + c] = v;
        if constexpr (F32) {
          const float wgt = bi < bj ? 2.0f : 1.0f;   // the mirror tile holds the same values
          const float p = wgt * v * v;
          const float e = wgt * fmaf(v, v, -v * v);
          const float tt = fs + p;
          const float bp = tt - fs;
          fc += (fs - (tt - bp)) + (p - bp) + e;
          fs = tt;
        } else {
          const double wgt = bi < bj ? 2.0 : 1.0;
          fd += wgt * v * v;
        }
        nbad += isfinite(v) ? 0 : 1;
        if (bi < bj) dst[(size_t)(bj * TS + rl) * Np + bi * TS + tx] = tile[tx][rl];
      }
      __syncthreads();
    }
    // partial sums of job m: Tr S0 (job 0) and ||S_m||_F^2
    double v[2] = {tr, F32 ? (double)fs + (double)fc : fd};
    block_sum<2, 256>(v, red);
    if (threadIdx.x == 0) {
      double* p = partials + ((size_t)m * ptiles + vb) * kNQ;
      p[kQTrace] = m == 0 ? v[0] : 0.0;
      p[kQFroNew] = v[1];
      p[kQFroDiff] = 0.0;
      p[kQBad] = 0.0;
    }
  }
  for (int m = m_lo > k ? m_lo : k + 1; m <= m_hi; ++m) {
    T* dst = master + (size_t)m * mat;
    for (int64_t idx = vb * blockDim.x + threadIdx.x; idx < (int64_t)mat;
         idx += vgrid * blockDim.x)
      dst[idx] = (T)0;
    if (threadIdx.x == 0) {
      double* p = partials + ((size_t)m * ptiles + vb) * kNQ;
      p[kQTrace] = 0.0;
      p[kQFroNew] = 0.0;
      p[kQFroDiff] = 0.0;
      p[kQBad] = 0.0;
    }
  }
  double vb_bad[1] = {(double)nbad};
  block_sum<1, 256>(vb_bad, red);
  if (threadIdx.x == 0) partials[((size_t)m_lo * ptiles + vb) * kNQ + kQBad] = vb_bad[0];
}

// One matrix per grid row: the matrices one after the other in each block was a
// chain of loads and block sums (n = 1000 k = 2 34 -> 21 us, order 3 at n = 512
// k = 2 19 -> 8 us; at n = 2048 k = 3 both take 46 us).
template <typename T>
__global__ void __launch_bounds__(256) init_kernel(State* st, T* master, const double* __restrict__ H,
                                                   const double* __restrict__ H1, int64_t n,
                                                   int64_t Np, int64_t ld, int k, int first_m,
                                                   const double* __restrict__ shift,
                                                   double* partials, int64_t ptiles) {
  pdl_wait();
  pdl_launch();
  const int m = first_m + (int)blockIdx.y;
  init_body<T>(st, master, H, H1, n, Np, ld, k, m, m, shift, partials, ptiles, blockIdx.x,
               gridDim.x);
}

int init_blocks(int64_t Np) {
  const int64_t tb = Np / kInitTile, pairs = tb * (tb + 1) / 2;
  return (int)(pairs < kInitBlocks ? pairs : kInitBlocks);
}

cudaError_t launch_init(const Layout& L, void* ws, const double* H, const double* H1,
                        int64_t ld, int k, int blocks, cudaStream_t s, int first_m,
                        const double* shift, int k_zero) {
  char* base = (char*)ws;
  State* st = (State*)(base + L.off_state);
  double* partials = (double*)(base + L.off_partials);
  const dim3 grid(blocks, k + k_zero + 1 - first_m);
  if (L.precision == DMPT_FP64)
    return launch_pdl(init_kernel<double>, grid, dim3(256), 0, s, st,
                      (double*)(base + L.off_master), H, H1, L.n, L.Np, ld, k, first_m, shift,
                      partials, L.partial_tiles);
  return launch_pdl(init_kernel<float>, grid, dim3(256), 0, s, st, (float*)(base + L.off_master),
                    H, H1, L.n, L.Np, ld, k, first_m, shift, partials, L.partial_tiles);
}

// ---------------------------------------------------------------------------
// Self-consistent response: charge potential and linear mixing of the
// induced charges q = diag(P1).

// v_j[r] = sum_c gamma[r][c] q_j[c]; one warp per row, FP64
__global__ void scc_potential_kernel(const double* __restrict__ gamma, int64_t n, int64_t ld,
                                     const double* __restrict__ q, double* v, int k) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r = warp; r < n; r += nw) {
    const double* g = gamma + r * ld;
    for (int j = 0; j < k; ++j) {
      const double* qj = q + (size_t)j * n;
      double acc = 0.0;
      for (int64_t c = lane; c < n; c += 32) acc = fma(g[c], qj[c], acc);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane == 0) v[(size_t)j * n + r] = acc;
    }
  }
}

cudaError_t launch_scc_potential(const double* gamma, int64_t n, int64_t ld, const double* q,
                                 double* v, int k, cudaStream_t s) {
  int64_t warps = n < 152 * 32 ? n : 152 * 32;
  scc_potential_kernel<<<(int)((warps * 32 + 255) / 256), 256, 0, s>>>(gamma, n, ld, q, v, k);
  return cudaGetLastError();
}

// one block per direction: red[j] = {||diag(P1_j) - q_j||^2, ||diag(P1_j)||^2}, then mix
__global__ void __launch_bounds__(256) scc_mix_kernel(const double* __restrict__ P1, int64_t n,
                                                      int64_t ld, double* q, double alpha,
                                                      double* red) {
  __shared__ double sm[2 * 256];
  const int j = blockIdx.x;
  const double* p = P1 + (size_t)j * n * ld;
  double* qj = q + (size_t)j * n;
  double d2 = 0.0, o2 = 0.0;
  for (int64_t r = threadIdx.x; r < n; r += 256) {
    const double qo = p[r * ld + r];
    const double d = qo - qj[r];
    d2 += d * d;
    o2 += qo * qo;
    qj[r] = (1.0 - alpha) * qj[r] + alpha * qo;
  }
  double v[2] = {d2, o2};
  block_sum<2, 256>(v, sm);
  if (threadIdx.x == 0) {
    red[4 * j + 0] = v[0];
    red[4 * j + 1] = v[1];
  }
}

cudaError_t launch_scc_mix(const double* P1, int64_t n, int64_t ld, double* q, int k,
                           double alpha, double* red, cudaStream_t s) {
  scc_mix_kernel<<<k, 256, 0, s>>>(P1, n, ld, q, alpha, red);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Device-side control (Alg. 1 branch rule, Alg. 2, Alg. 3).

__device__ int fp16_exponent_for(double bound) {
  // exponent e with bound * 2^e < 2^kFp16TargetExp
  if (!(bound > 0.0) || !isfinite(bound)) return 0;
  int e = kFp16TargetExp - (ilogb(bound) + 1);
  return e < -100 ? -100 : (e > 100 ? 100 : e);
}

// A decide step works on the control block's head (every field before the
// per-layer histories) in shared memory.  What bounds it is latency, not work:
// one thread walking the block in device memory took 9-35 us per layer (a
// dependent access costs about 0.4 us, an FP64 square root or divide as much).
// Here the head and the few history entries the tests read are fetched while
// the layer product still runs, the partial sums of four jobs are added at once
// by 256 threads each, their square roots are taken in parallel, and one warp
// then takes the decisions, lane j those of response slot j.  Measured from the
// end of the layer to the end of the step, n = 128 k = 1: 16.5 us by one
// thread, 4.0 us with every read after the layer's end and a 256-wide FP64
// tree per quantity, 3.0 us now.
constexpr int kDecideThreads = 1024;
static_assert(kHeadWords <= kDecideThreads, "one head word per thread");

struct DecideShared {
  alignas(16) unsigned head[kHeadWords + (kHeadWords & 1)];
  double red[kDecideThreads / 256][8][kNQ];
  double sums[kMaxK + 1][kNQ];   // per job, as summed from the partials
  double roots[kMaxK + 1][kNQ];  // their square roots, taken in parallel
  double fe2[kMaxK];             // FroErr^(1)_{n-2} of the layer that has run
  double iderr1;                 // IdErr_{n-1}
  int sig0, sig1, sig_next;      // sigma_n, sigma_{n-1}; sigma of the layer to plan
};

// Plan layer n (Alg. 1: branch choice; Alg. 2: D0 stopping tests).  One warp;
// S: head in shared memory, G: control block, conv: slot `lane` has stopped.
// root: sqrt(s1_fro2) of slot `lane`.
__device__ void plan_layer(State* S, State* G, const DecideShared& sh, int n, int lane,
                           bool conv, double root) {
  if (lane == 0) {
    int sigma;
    if (!S->d0_conv) {
      const double NS = S->NS, NX = S->NX, no = S->n_occ;
      const double iderr = NS - NX;
      // sigma_n = sign(|2 N_S - N_X - N_occ| - |N_X - N_occ|); sign(0) -> -1
      const double arg = fabs(2.0 * NS - NX - no) - fabs(NX - no);
      sigma = arg > 0.0 ? 1 : -1;
      G->iderr[n] = iderr;
      G->ns_hist[n] = NS;
      G->nx_hist[n] = NX;
      bool stop = iderr <= 0.0;
      if (!stop && n > 2 && sh.sig0 != sh.sig1 && iderr > S->c_d0 * sh.iderr1 * sh.iderr1)
        stop = true;
      S->plan_square = 1;
      if (stop) {
        S->d0_conv = 1;
        S->d0_layer = n;
        S->plan_write0 = 0;  // this layer's square only measures FroErr^(0)
      } else {
        S->plan_write0 = 1;
      }
    } else {
      sigma = -sh.sig0;  // the sigma flip of Alg. 1
      S->plan_square = 0;
      S->plan_write0 = 0;
    }
    G->sigma[n] = (signed char)sigma;
    S->sigma_cur = sigma;
    S->n_layer = n;
  }
  __syncwarp();   // s1_fro2 of every slot
  if (lane < S->k) {
    S->plan_resp[lane] = !conv;
    // |S1_n|_max <= ||S1_n||_2 <= (2 ||S0||_2 + |1 - sigma|) ||S1_{n-1}||_2
    //            <= 4.5 ||S1_{n-1}||_F   (spectrum of S0 within [-0.25, 1.25]);
    // an order-o slot (o >= 2) adds sum_{a=1}^{o-1} ||S_a S_{o-a}||_2
    // <= sum ||S_a||_F ||S_{o-a}||_F (twice, for 2 S - S^2)
    double bound = 4.5 * root;
    if (S->order >= 2 && lane >= S->k1) {
      const int o = 1 + lane / S->k1, d = lane % S->k1;
      double cross = 0.0;
      for (int a = 1; a < o; ++a)
        cross += sqrt(S->s1_fro2[(a - 1) * S->k1 + d] * S->s1_fro2[(o - a - 1) * S->k1 + d]);
      bound += 2.0 * cross;
    }
    S->s1_exp_next[lane] = S->precision == DMPT_DUAL_FP16 ? fp16_exponent_for(bound) : 0;
  }
}

// Plan layer m of a response replay: S0 operand = stored state
// min(m - 1, U), the forward's sigma_m (continued by flips past the forward's
// last layer), responses of the directions still running.
__device__ void plan_replay(State* S, State* G, const DecideShared& sh, int m, int lane,
                            bool conv, double root) {
  if (lane == 0) {
    const int U = S->d0_updates;
    S->z0_cur = S->tape_base + 2 * (m - 1 < U ? m - 1 : U);
    int sigma = sh.sig_next;
    if (m > S->rp_lmax) {
      sigma = -sh.sig0;
      G->sigma[m] = (signed char)sigma;
    }
    S->sigma_cur = sigma;
    S->plan_square = 0;
    S->plan_write0 = 0;
    S->n_layer = m;
  }
  if (lane < S->k) {
    S->plan_resp[lane] = !conv;
    S->s1_exp_next[lane] =
        S->precision == DMPT_DUAL_FP16 ? fp16_exponent_for(4.5 * root) : 0;
  }
}

// End of a run (lane 0).
__device__ __forceinline__ void decide_end(State* S, int lane, int status) {
  if (lane == 0) {
    S->status = status;
    S->done = 1;
  }
}

// Response replayed over the stored S0 states (one warp).
__device__ void decide_replay(State* S, State* G, const DecideShared& sh, int mode, int lane) {
  const bool init = mode == kDecideReplayInit;
  const int k = S->k, n = S->n_layer;
  const bool ran = lane < k && (init || S->plan_resp[lane]);
  const bool bad = __any_sync(0xffffffffu, ran && sh.sums[1 + (ran ? lane : 0)][kQBad] > 0.0);
  if (S->timeout_flag) return decide_end(S, lane, DMPT_ETIMEOUT);
  if (bad) return decide_end(S, lane, DMPT_ENUMERIC);
  bool conv = true;
  double root = 0.0;   // sqrt(s1_fro2) of this lane's slot
  if (init) {
    if (lane < k) {
      S->cur1[lane] = 0;
      S->d1_conv[lane] = 0;
      S->d1_layer[lane] = 0;
      const double f = sh.sums[1 + lane][kQFroNew];
      S->s1_fro2[lane] = f;
      root = sh.roots[1 + lane][kQFroNew];
      S->s1_exp_cur[lane] = S->precision == DMPT_DUAL_FP16 ? fp16_exponent_for(root) : 0;
      conv = false;
    }
    if (lane == 0) {
      S->rp_lmax = S->layers_run;
      S->rp_layers = 0;
    }
    __syncwarp();
    return plan_replay(S, G, sh, 1, lane, conv, root);
  }
  if (lane < k) conv = S->d1_conv[lane] != 0;
  if (ran) {
    const double fe = sh.roots[1 + lane][kQFroDiff];
    G->froerr1[lane][n] = fe;
    const bool fired = n - 2 >= S->d0_layer && fe >= S->c_pt * S->froerr0 * sh.fe2[lane];
    if (fired) {
      S->d1_conv[lane] = 1;
      S->d1_layer[lane] = n;
      conv = true;
    } else {
      S->cur1[lane] ^= 1;
      S->s1_fro2[lane] = sh.sums[1 + lane][kQFroNew];
      root = sh.roots[1 + lane][kQFroNew];
      S->s1_exp_cur[lane] = S->s1_exp_next[lane];
    }
  }
  if (lane < k && conv) root = sqrt(S->s1_fro2[lane]);
  if (lane == 0) S->rp_layers = n;
  const bool all1 = __all_sync(0xffffffffu, conv);
  if (all1) return decide_end(S, lane, DMPT_OK);
  if (n + 1 > S->max_layers) return decide_end(S, lane, DMPT_ENOTCONV);
  plan_replay(S, G, sh, n + 1, lane, conv, root);
}

// Adjoint of the S0 recursion, run backwards over the stored states (lane 0).
__device__ void decide_adjoint(State* S, const DecideShared& sh, int mode) {
  if (S->timeout_flag) return decide_end(S, 0, DMPT_ETIMEOUT);
  if (mode != kDecideAdjResume && sh.sums[1][kQBad] > 0.0) return decide_end(S, 0, DMPT_ENUMERIC);
  int m;
  if (mode == kDecideAdjInit) {
    S->k = 1;
    S->cur1[0] = 0;
    S->plan_square = 0;
    S->plan_write0 = 0;
    for (int j = 0; j < kMaxK; ++j) S->plan_resp[j] = 0;
    S->s1_fro2[0] = sh.sums[1][kQFroNew];
    S->s1_exp_cur[0] =
        S->precision == DMPT_DUAL_FP16 ? fp16_exponent_for(sqrt(S->s1_fro2[0])) : 0;
    m = S->d0_updates;
  } else if (mode == kDecideAdjLayer) {
    S->cur1[0] ^= 1;
    S->s1_fro2[0] = sh.sums[1][kQFroNew];
    S->s1_exp_cur[0] = S->s1_exp_next[0];
    m = S->adj_m - 1;
  } else {
    m = S->adj_m;   // resume after the host reloaded the tape with an earlier segment
  }
  S->adj_m = m;
  if (m <= 0) {
    S->plan_resp[0] = 0;
    return decide_end(S, 0, DMPT_OK);
  }
  if (m <= S->adj_seg_a) {
    // S_{m-1} lies before the states in the tape (checkpointed run): the
    // host recomputes the previous segment and resumes with layer m
    S->plan_resp[0] = 0;
    return;
  }
  // adjoint of layer m: Gbar <- sigma_m (S_{m-1} Gbar + Gbar S_{m-1}) + (1 - sigma_m) Gbar
  // (the tape holds states adj_seg_a, adj_seg_a + 1, ...; 0 without checkpoints)
  S->z0_cur = S->tape_base + 2 * (m - 1 - S->adj_seg_a);
  S->sigma_cur = sh.sig_next;   // sigma_m
  S->plan_resp[0] = 1;
  S->s1_exp_next[0] = S->precision == DMPT_DUAL_FP16
                          ? fp16_exponent_for(4.5 * sqrt(S->s1_fro2[0]))
                          : 0;
}

// The initial layer has run: start of a forward run (one warp).
__device__ void decide_init(State* S, State* G, const DecideShared& sh, int lane) {
  const bool bad =
      __any_sync(0xffffffffu, lane <= S->k && sh.sums[lane <= S->k ? lane : 0][kQBad] > 0.0);
  if (!(S->epsN > S->eps1) || !isfinite(S->epsN) || !isfinite(S->eps1) || bad)
    return decide_end(S, lane, DMPT_ENUMERIC);
  if (lane == 0) {
    S->NS = sh.sums[0][kQTrace];
    S->NX = sh.sums[0][kQFroNew];
    S->s0_exp = S->precision == DMPT_DUAL_FP16 ? kFp16TargetExp - 1 : 0;
    S->cur0 = 0;
    S->d0_updates = 0;
    S->ckpt_pending = S->ckpt_k >= 2 ? 1 : 0;   // S_0 is checkpoint 0
    S->z0_cur = S->tape ? S->tape_base : zslice(0, 0, 0, S->layout_k);
    S->z0_next = S->tape ? S->tape_base + 2 : zslice(1, 0, 0, S->layout_k);
    S->d0_conv = 0;
    S->d0_layer = 0;
    S->layers_run = 0;
    S->froerr0 = 0.0;
  }
  double root = 0.0;
  if (lane < S->k) {
    S->cur1[lane] = 0;
    S->d1_conv[lane] = 0;
    S->d1_layer[lane] = 0;
    S->s1_fro2[lane] = sh.sums[1 + lane][kQFroNew];
    root = sh.roots[1 + lane][kQFroNew];
    S->s1_exp_cur[lane] = S->precision == DMPT_DUAL_FP16 ? fp16_exponent_for(root) : 0;
  }
  __syncwarp();
  plan_layer(S, G, sh, 1, lane, false, root);
}

// A layer product has finished: apply its results (one warp).
__device__ void decide_layer(State* S, State* G, const DecideShared& sh, int lane) {
  const int k = S->k, n = S->n_layer;
  const bool square = S->plan_square != 0, wrote = S->plan_write0 != 0;
  const bool d0 = S->d0_conv != 0;
  const bool ran = lane < k && S->plan_resp[lane];
  bool bad = __any_sync(0xffffffffu, ran && sh.sums[1 + (ran ? lane : 0)][kQBad] > 0.0);
  bad = bad || (square && sh.sums[0][kQBad] > 0.0);
  if (S->timeout_flag) return decide_end(S, lane, DMPT_ETIMEOUT);
  if (bad) return decide_end(S, lane, DMPT_ENUMERIC);
  bool conv = lane < k ? S->d1_conv[lane] != 0 : true;
  double root = 0.0;   // sqrt(s1_fro2) of this lane's slot
  if (square && lane == 0) {
    if (wrote) {
      S->NS = sh.sums[0][kQTrace];    // Tr S_n      (N_S of Alg. 2)
      S->NX = sh.sums[0][kQFroNew];   // ||S_n||_F^2 = Tr S_n^2 (N_X of the next layer)
      S->cur0 ^= 1;
      S->d0_updates += 1;
      if (S->ckpt_k >= 2 && S->d0_updates % S->ckpt_k == 0) S->ckpt_pending = 1;
      if (S->tape) {
        S->z0_cur = S->z0_next;
        S->z0_next += 2;
      } else {
        S->z0_cur = zslice(S->cur0, 0, 0, S->layout_k);
        S->z0_next = zslice(S->cur0 ^ 1, 0, 0, S->layout_k);
      }
    } else {
      S->froerr0 = sh.roots[0][kQFroDiff];  // FroErr^(0) of Alg. 2
    }
  }
  __syncwarp();
  if (ran) {
    const double fe = sh.roots[1 + lane][kQFroDiff];  // FroErr^(1)_n of Alg. 3
    G->froerr1[lane][n] = fe;
    bool fired = false;
    if (d0 && n - 2 >= S->d0_layer) fired = fe >= S->c_pt * S->froerr0 * sh.fe2[lane];
    if (fired) {
      S->d1_conv[lane] = 1;  // keep S1_{n-1}: the buffer written by this layer is dropped
      S->d1_layer[lane] = n;
      conv = true;
    } else {
      S->cur1[lane] ^= 1;
      S->s1_fro2[lane] = sh.sums[1 + lane][kQFroNew];
      root = sh.roots[1 + lane][kQFroNew];
      S->s1_exp_cur[lane] = S->s1_exp_next[lane];
    }
  }
  if (lane < k && conv) root = sqrt(S->s1_fro2[lane]);
  if (lane == 0) S->layers_run = n;
  const bool all1 = __all_sync(0xffffffffu, conv);
  const bool end = d0 && all1, cap = n + 1 > S->max_layers;
  if (end || cap) {
    if (lane == 0) S->n_layer = n + 1;
    return decide_end(S, lane, end ? DMPT_OK : DMPT_ENOTCONV);
  }
  plan_layer(S, G, sh, n + 1, lane, conv, root);
}

// The decide step of one instance, run by one block of kDecideThreads
// threads.  jobs: 1 + the response slots of the partials array.
// Pdl: launched while the kernel before it may still run.  That kernel is a
// layer product or an initial kernel, which write nothing of the control block
// but timeout_flag (and round_ctr, reset here), and it started after the last
// kernel that did write the block had finished, so the rest is read before
// pdl_wait().  The exception is kDecideAdjResume, which follows the step kernel
// between recompute layers or the load of a segment: a grid's writes are only
// visible after the wait (its end alone, without pdl_launch(), orders nothing),
// and the whole head is stored back below, so it waits first.
template <bool Pdl>
__device__ void decide_body(State* st, const double* partials, int64_t ptiles,
                            int64_t entries, int jobs, int mode, DecideShared& sh,
                            const int* group_timeout = nullptr) {
  const int tid = threadIdx.x, lane = tid & 31;
  if constexpr (Pdl) {
    if (mode == kDecideAdjResume) pdl_wait();
  }
  if (tid < kHeadWords) sh.head[tid] = __ldcg(reinterpret_cast<const unsigned*>(st) + tid);
  if (tid >= kDecideThreads - 32) {
    // the history entries the tests read, fetched while the sums are formed
    const bool adj = mode == kDecideAdjInit || mode == kDecideAdjLayer || mode == kDecideAdjResume;
    const bool fresh = mode == kDecideInit || mode == kDecideReplayInit;
    const int n = fresh ? 0 : __ldcg(&st->n_layer);   // the layer that has run
    if (lane < kMaxK && !adj && n >= 2) sh.fe2[lane] = __ldcg(&st->froerr1[lane][n - 2]);
    if (lane == 8 && !adj && n >= 1) sh.iderr1 = __ldcg(&st->iderr[n - 1]);
    if (lane == 9 && !adj) sh.sig0 = __ldcg(&st->sigma[n]);
    if (lane == 10 && !adj && n >= 1) sh.sig1 = __ldcg(&st->sigma[n - 1]);
    if (lane == 11) {
      int m = n + 1;
      if (adj)
        m = mode == kDecideAdjInit
                ? __ldcg(&st->d0_updates)
                : __ldcg(&st->adj_m) - (mode == kDecideAdjLayer ? 1 : 0);
      sh.sig_next = m >= 0 && m <= kMaxL ? __ldcg(&st->sigma[m]) : 0;
    }
  }
  if constexpr (Pdl) {
    pdl_wait();
    constexpr int kTimeoutWord = (int)(offsetof(State, timeout_flag) / sizeof(unsigned));
    if (tid == kTimeoutWord)
      sh.head[tid] = group_timeout && __ldcg(group_timeout)
                         ? 1u
                         : __ldcg(reinterpret_cast<const unsigned*>(st) + tid);
  }
  // Sums of the partials, four jobs at once, in a fixed order: lane 4 u + q of
  // warp w of a job adds quantity q of the entries 8 w + u (mod 64), three
  // shuffles add a warp's eight, and one warp adds the job's eight warps and
  // takes the square roots.  The part runs two FP64 operations per clock and
  // SM, so a warp's addition holds the pipe for 16 clocks: their number counts.
  const int grp = tid >> 8, w = (tid >> 5) & 7, q = lane & 3;
  for (int j0 = 0; j0 < jobs; j0 += kDecideThreads / 256) {
    const int job = j0 + grp;
    if (job < jobs) {
      double v = 0.0;
      const double* p = partials + ((size_t)job * ptiles + 8 * w + (lane >> 2)) * kNQ + q;
#pragma unroll 4
      for (int64_t e = 8 * w + (lane >> 2); e < entries; e += 64, p += 64 * kNQ) v += __ldcg(p);
      if (8 * w < entries) {
#pragma unroll
        for (int o = 16; o >= 4; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
      }
      if (lane < 4) sh.red[grp][w][lane] = v;
    }
    __syncthreads();
    if (job < jobs && w == 0) {
      double x = sh.red[grp][lane >> 2][q];
#pragma unroll
      for (int o = 16; o >= 4; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
      if (lane < 4) {
        sh.sums[job][lane] = x;
        sh.roots[job][lane] = sqrt(x);
      }
    }
    __syncthreads();
  }
  State* S = reinterpret_cast<State*>(sh.head);   // only the fields before the histories
  if (tid < 32) {
    if (lane == 0) {
      S->round_ctr = 0u;    // for the next pair-kernel launch
      S->ckpt_pending = 0;  // set again below when this step makes a checkpointed state
    }
    __syncwarp();
    if (!S->done) {
      switch (mode) {
        case kDecideInit: decide_init(S, st, sh, lane); break;
        case kDecideLayer: decide_layer(S, st, sh, lane); break;
        case kDecideReplayInit:
        case kDecideReplayLayer: decide_replay(S, st, sh, mode, lane); break;
        default:
          if (lane == 0) decide_adjoint(S, sh, mode);
      }
    }
  }
  __syncthreads();
  if (tid < kHeadWords) reinterpret_cast<unsigned*>(st)[tid] = sh.head[tid];
}

__global__ void __launch_bounds__(kDecideThreads)
    decide_kernel(State* st, const double* partials, int64_t ptiles, int64_t entries,
                  int jobs, int mode, volatile unsigned* progress, unsigned code) {
  __shared__ DecideShared sh;
  pdl_launch();
  decide_body<true>(st, partials, ptiles, entries, jobs, mode, sh);
  if (progress && threadIdx.x == 0)
    *progress = code | (reinterpret_cast<const State*>(sh.head)->done ? 1u : 0u);
}

// Layer decide of every instance of a grouped launch, one block each; the last
// block to finish reports to the host (progress, as in decide_kernel; bit 0:
// every instance has ended).
__global__ void __launch_bounds__(kDecideThreads)
    decide_group_kernel(const GroupDecide* __restrict__ args, const int* group_timeout,
                        GroupQueue* queue, volatile unsigned* progress, unsigned code) {
  __shared__ DecideShared sh;
  pdl_launch();
  const GroupDecide a = args[blockIdx.x];
  decide_body<true>(a.st, a.partials, a.ptiles, a.entries, a.jobs, kDecideLayer, sh,
                    group_timeout);
  if (threadIdx.x != 0) return;
  if (blockIdx.x == 0) {   // the next grouped launch starts a new queue
    queue->counter = 0u;
    queue->epoch += 1u;
  }
  // blocks that are through (low half) and instances that have ended (high half)
  const unsigned one = 1u | (reinterpret_cast<const State*>(sh.head)->done ? 0x10000u : 0u);
  const unsigned all = atomicAdd(&queue->decided, one) + one;
  if ((all & 0xFFFFu) == gridDim.x) {
    queue->decided = 0u;
    *progress = code | ((all >> 16) == gridDim.x ? 1u : 0u);
  }
}

cudaError_t launch_decide_group(const GroupDecide* args, int count, const int* group_timeout,
                                GroupQueue* queue, unsigned* progress, unsigned code,
                                cudaStream_t s) {
  if (count < 1) return cudaSuccess;
  return launch_pdl(decide_group_kernel, dim3(count), dim3(kDecideThreads), 0, s, args,
                    group_timeout, queue, progress, code);
}

// Per-device one-time setup; thread-safe.  The decide kernel runs between
// layer kernels that use nearly all of an SM's shared memory: with the same
// split of L1 and shared memory the SM need not be reconfigured.
static void decide_setup() {
  constexpr int kDevices = 64;
  static std::once_flag once[kDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) return;
  std::call_once(once[dev], [] {
    cudaFuncSetAttribute(decide_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                         cudaSharedmemCarveoutMaxShared);
  });
}

cudaError_t launch_decide(const Layout& L, void* ws, int mode, int64_t entries, cudaStream_t s,
                          unsigned* progress, unsigned code) {
  char* base = (char*)ws;
  decide_setup();
  return launch_pdl(decide_kernel, dim3(1), dim3(kDecideThreads), 0, s,
                    (State*)(base + L.off_state), (const double*)(base + L.off_partials),
                    L.partial_tiles, entries, 1 + L.k, mode, progress, code);
}

// ---------------------------------------------------------------------------
// FP32 layer product with fused epilogue.
//
// Grid: (upper tiles, 1 + slots).  Job 0 computes X = S0 S0 (Sec. II B,
// Eq. (DNN-SP2_act)) for tile (I, J), I <= J; job 1+k computes
// X1 = S0 S1_k + S1_k S0 (activation f^(1), Eq. (eq:activation-function))
// as one accumulation over two K-passes; a higher-order term (Sec. III A,
// Eq. (S_n detailed)) adds its cross products S_a S_{o-a} as further passes.
// Both operands are read as row
// panels: for symmetric B, B[k][j] = B[j][k].  The epilogue applies
// S_n = sigma X + (1 - sigma) S_{n-1} (Eq. (eq:Sn); Alg. 2 / Alg. 3 updates)
// to the elements with row <= col, stores them at (r, c) and (c, r) in the
// other ping-pong buffer, and reduces the Alg. 2 / 3 norms in FP64.

template <int TM>
__device__ __forceinline__ int frag_index(int t, int m) {
  // the TM rows (cols) of a thread: two runs of TM/2 contiguous elements,
  // the second BT/2 after the first
  constexpr int H = TM / 2;
  constexpr int BT = 16 * TM;
  return m < H ? t * H + m : BT / 2 + t * H + (m - H);
}

// Jobs of a layer (as in the tensor-core kernels): 0 = square of S0; job
// 1 + (o - 1) k1 + d = the order-o term of direction d, in o + 1 K passes
// (pass 0 = S0 S_o, pass 1 = S_o S0, pass p >= 2 = S_{p-1} S_{o-p+1}).
__device__ __forceinline__ int simt_job_order(int job, int k1) { return 1 + (job - 1) / k1; }
__device__ __forceinline__ int simt_job_passes(int job, int k1) {
  return job == 0 ? 1 : (job <= k1 ? 2 : 1 + simt_job_order(job, k1));
}
__device__ __forceinline__ int simt_job_slot(int job, int a, int k1) {
  return 1 + (a - 1) * k1 + (job - 1) % k1;
}
__device__ __forceinline__ void simt_job_operands(int job, int pass, int k1, int* mA, int* mB) {
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
    *mA = simt_job_slot(job, pass - 1, k1);
    *mB = simt_job_slot(job, simt_job_order(job, k1) - pass + 1, k1);
  }
}

// 16-byte asynchronous copy global -> shared (L2 only), and its group waits
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(smem)),
               "l"(gmem)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Shared memory of the SIMT layer kernel: SIMT_STAGES stages of the two
// operand slabs (BK x BT, rows padded by one 16-byte chunk), then the
// block's reduction array.
constexpr int SIMT_STAGES = 3;
template <int TM, int BK>
constexpr int simt_smem_bytes() {
  return SIMT_STAGES * 2 * BK * (16 * TM + 4) * (int)sizeof(float) + 4 * 256 * 8;
}

template <int TM, int BK>
__global__ void __launch_bounds__(256, TM == 8 ? 2 : 4)
    layer_simt_kernel(State* st, float* __restrict__ master, int64_t n, int64_t Np, int k,
                      double* __restrict__ partials, int64_t ptiles) {
  constexpr int BT = 16 * TM;
  constexpr int VW = 4;                        // elements per 16-byte copy
  constexpr int LD = BT + VW;                  // padded row of a slab
  constexpr int CPR = BT / VW;                 // copies per slab row
  constexpr int NCP = BK * CPR / 256;          // copies per thread per slab
  static_assert(NCP >= 1 && (BK * CPR) % 256 == 0, "slab copies divide over the block");

  // stage s: As = slab of the A operand, Bs = slab of the B operand, each
  // BK rows (K index) x BT columns (output rows / columns of the tile)
  extern __shared__ __align__(16) uint8_t simt_smem[];
  float* slabs = reinterpret_cast<float*>(simt_smem);
  double* red = reinterpret_cast<double*>(simt_smem + SIMT_STAGES * 2 * BK * LD * sizeof(float));

  pdl_wait();   // no pdl_launch(): see layer_fp64_kernel
  if (st->done) return;
  const int job = (int)gridDim.y - 1 - (int)blockIdx.y;   // most K passes first
  const int run = job == 0 ? st->plan_square : st->plan_resp[job - 1];
  if (!run) return;

  // upper tile (I, J), I <= J, row-major over the upper triangle of the tiles
  // that hold elements of the n x n matrix
  const int T_ = (int)((n + BT - 1) / BT);
  int64_t t = blockIdx.x;
  int I = 0;
  while (t >= T_ - I) {
    t -= T_ - I;
    ++I;
  }
  const int J = I + (int)t;

  const size_t mat = (size_t)Np * Np;
  const int cur0 = st->cur0;
  const int cur = job == 0 ? cur0 : st->cur1[job - 1];
  const float* Sj = master + (size_t)(cur * (1 + k) + job) * mat;   // the job's own slot
  float* out = master + (size_t)((cur ^ 1) * (1 + k) + job) * mat;

  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  // column pairs (2 j, 2 j + 1) of the thread's tile, packed: one product per
  // FMA fills the issue slots, and the shared-memory reads come on top.  n = 4096
  // k = 1 layer 3.80 -> 3.53 ms.  While an SM has blocks its FMA pipe is active in
  // 80% of the cycles (four warps per scheduler, which at times all wait for
  // operand reads or the barrier of a K step), and at n = 4096 the SMs have
  // blocks for 95% of the layer (n = 2560: 78% and 83%).
  f32x2 acc2[TM][TM / 2];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM / 2; ++j) acc2[i][j] = pack2(0.0f, 0.0f);

  const int k1 = st->order >= 2 ? st->k1 : k;   // first-order directions
  const int passes = simt_job_passes(job, k1);
  const int nkb = (int)((n + BK - 1) / BK);   // the K range of the padding is zero
  for (int pass = 0; pass < passes; ++pass) {
    // pass p of the job: A = slot mA rows I, B = slot mB rows J (square:
    // S0 S0; order-o term: S0 S_o, S_o S0, then S_{p-1} S_{o-p+1}).  The
    // masters are exactly symmetric (both halves are always written with the
    // same value), so the K x BT slab A[I rows][kb ..] is read as rows
    // kb .. kb + BK - 1, columns I BT .. I BT + BT - 1: contiguous 16-byte
    // copies that land in shared memory already K-major.
    int mA, mB;
    simt_job_operands(job, pass, k1, &mA, &mB);
    const float* A = master + (size_t)((mA == 0 ? cur0 : st->cur1[mA - 1]) * (1 + k) + mA) * mat +
                 (size_t)I * BT;
    const float* B = master + (size_t)((mB == 0 ? cur0 : st->cur1[mB - 1]) * (1 + k) + mB) * mat +
                 (size_t)J * BT;
    auto load = [&](int stage, int kb) {
      float* as = slabs + (size_t)stage * 2 * BK * LD;
      float* bs = as + BK * LD;
#pragma unroll
      for (int v = 0; v < NCP; ++v) {
        const int idx = tid + 256 * v;
        const int row = idx / CPR, cq = idx % CPR;
        const size_t g = (size_t)(kb + row) * Np + cq * VW;
        cp_async16(as + row * LD + cq * VW, A + g);
        cp_async16(bs + row * LD + cq * VW, B + g);
      }
    };
    __syncthreads();   // every stage of the previous pass has been read
    // prologue: stages 0 .. SIMT_STAGES - 2 in flight (one group each)
#pragma unroll
    for (int sidx = 0; sidx < SIMT_STAGES - 1; ++sidx) {
      if (sidx < nkb) load(sidx, sidx * BK);
      cp_async_commit();
    }
    for (int it = 0; it < nkb; ++it) {
      cp_async_wait<SIMT_STAGES - 2>();   // stage it has landed (this thread's copies)
      __syncthreads();                    // ... and every thread's; stage it - 1 is free
      {
        const int nx = it + SIMT_STAGES - 1;
        if (nx < nkb) load(nx % SIMT_STAGES, nx * BK);
        cp_async_commit();
      }
      const float* as = slabs + (size_t)(it % SIMT_STAGES) * 2 * BK * LD;
      const float* bs = as + BK * LD;
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) {
        float a[TM];
        f32x2 b[TM / 2];
#pragma unroll
        for (int m = 0; m < TM; ++m) a[m] = as[kk * LD + frag_index<TM>(ty, m)];
        if constexpr (TM == 8) {
#pragma unroll
          for (int m = 0; m < TM / 2; m += 2) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(
                bs + kk * LD + frag_index<TM>(tx, 2 * m));
            b[m] = v.x;
            b[m + 1] = v.y;
          }
        } else {
#pragma unroll
          for (int m = 0; m < TM / 2; ++m)
            b[m] = *reinterpret_cast<const f32x2*>(bs + kk * LD + frag_index<TM>(tx, 2 * m));
        }
#pragma unroll
        for (int i = 0; i < TM; ++i) {
          const f32x2 ai = pack2(a[i], a[i]);
#pragma unroll
          for (int j = 0; j < TM / 2; ++j) acc2[i][j] = fma2(ai, b[j], acc2[i][j]);
        }
      }
    }
    cp_async_wait<0>();   // no copy of this pass left in flight
  }

  // ---- fused epilogue
  const float sg = (float)st->sigma_cur;
  const float om = 1.0f - sg;
  const bool write = job == 0 ? st->plan_write0 != 0 : true;
  double tr = 0.0, bad = 0.0;
  // ||S_new||_F^2 and ||S_old - X||_F^2 as exact FP32 products summed with
  // TwoSum compensation (the FP64 rate of the part is low), converted to FP64
  // once per thread
  float fn_s = 0.0f, fn_c = 0.0f, fd_s = 0.0f, fd_c = 0.0f;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int64_t r = (int64_t)I * BT + frag_index<TM>(ty, i);
#pragma unroll
    for (int j = 0; j < TM; ++j) {
      const int64_t c = (int64_t)J * BT + frag_index<TM>(tx, j);
      if (r > c) continue;  // owned by the mirrored element
      float x01[2];
      unpack2(acc2[i][j / 2], x01[0], x01[1]);
      const float x = x01[j % 2];
      const float old = Sj[(size_t)r * Np + c];
      if (!isfinite(x)) bad += 1.0;
      const float nw = sg * x + om * old;
      const float w = (r == c) ? 1.0f : 2.0f;
      const float dd = old - x;
      {
        const float p = w * dd * dd;
        const float e = w * fmaf(dd, dd, -dd * dd);
        const float tt = fd_s + p;
        const float bp = tt - fd_s;
        fd_c += (fd_s - (tt - bp)) + (p - bp) + e;
        fd_s = tt;
      }
      if (write) {
        const float p = w * nw * nw;
        const float e = w * fmaf(nw, nw, -nw * nw);
        const float tt = fn_s + p;
        const float bp = tt - fn_s;
        fn_c += (fn_s - (tt - bp)) + (p - bp) + e;
        fn_s = tt;
      }
      if (write) {
        out[(size_t)r * Np + c] = nw;
        if (r != c) out[(size_t)c * Np + r] = nw;
        if (r == c) tr += (double)nw;
      }
    }
  }
  const double fnew = (double)fn_s + (double)fn_c;
  const double fdiff = (double)fd_s + (double)fd_c;
  double v[4] = {tr, fnew, fdiff, bad};
  block_sum<4, 256>(v, red);
  if (tid == 0) {
    double* p = partials + ((size_t)job * ptiles + blockIdx.x) * kNQ;
#pragma unroll
    for (int q = 0; q < 4; ++q) p[q] = v[q];
  }
}

// ---------------------------------------------------------------------------
// FP64 layer product with fused epilogue.
//
// The part runs two FP64 FMAs per clock and SM, so a warp's FMA holds the
// SM's pipe for 16 clocks and everything else (shared-memory reads, copies,
// indexing) hides behind it: what counts is that every SM gets the same
// number of them and that none is spent on padding.  So the tiles are small
// (FP64_TILE below), run over the n x n matrix rather than its padding to
// 256, and a block is four warps that each sum a quarter of the K range of the
// whole tile (k = w mod 4); the quarters are added in a fixed order.  Blocks
// of the jobs with the most K passes start first.  Elements outside n x n are
// neither computed on nor written: rows of the K range beyond n are filled
// with zeros on the way to shared memory, and what a tile's columns beyond n
// hold reaches discarded elements only.
// Measured per layer, one direction (64 x 64 tiles over the padded matrix,
// one thread per 4 x 4 elements -> now): n = 128
// 531 -> 12.9 us, n = 700 2326 -> 939 us (0.82 ms at two FMAs per clock and
// SM).
//
// Tile edge: 8 up to n = 400, where 16 leaves SMs with a tile more than
// others; 16 up to n = 2048; 32 above, where the balance no longer depends on
// it and larger tiles keep the partial sums few.
// 16-byte asynchronous copy that writes zeros instead when `in` is false
__device__ __forceinline__ void cp_async16_zfill(void* smem, const void* gmem, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(smem)),
               "l"(gmem), "r"(in ? 16 : 0)
               : "memory");
}

template <int T>
__global__ void __launch_bounds__(128)
    layer_fp64_kernel(const State* st, double* master, int64_t n,
                      int64_t Np, int k, double* __restrict__ partials, int64_t ptiles) {
  constexpr int BK = 16, STAGES = 3, NT = 128;
  constexpr int LD = T + 2;                 // padded slab row (16-byte chunks)
  constexpr int RA = T / 8, CB = T / 4;     // a lane's rows and columns of the tile
  constexpr int NCP = BK * T / NT;          // 16-byte copies per thread and stage (A and B)
  constexpr int NE = (T * T + NT - 1) / NT; // elements per thread in the epilogue
  constexpr int SLAB = BK * LD;
  constexpr int SMEM = STAGES * 2 * SLAB > 4 * T * T ? STAGES * 2 * SLAB : 4 * T * T;
  // the copy stages; after the K loop the four warps' sums, then the new tile
  __shared__ __align__(16) double sm[SMEM];
  __shared__ double red[2][NT];
  __shared__ double red_tr[32];

  // The next kernel starts when this one's blocks have all ended (no
  // pdl_launch() here): blocks of the next layer that come in while this one's
  // last blocks run would fill the SMs that ended first and leave the layer
  // unbalanced (FP64 form, n = 700: 39.1 ms against 37.2).
  pdl_wait();
  if (st->done) return;
  const int job = (int)gridDim.y - 1 - (int)blockIdx.y;
  const bool run = job == 0 ? st->plan_square != 0 : st->plan_resp[job - 1] != 0;
  if (!run) return;

  // upper tile (I, J), I <= J: blockIdx.x = J (J + 1) / 2 + I
  const int64_t t = blockIdx.x;
  int64_t J = (int64_t)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while ((J + 1) * (J + 2) / 2 <= t) ++J;
  while (J * (J + 1) / 2 > t) --J;
  const int64_t I = t - J * (J + 1) / 2;
  const bool diag = I == J;

  const size_t mat = (size_t)Np * Np;
  const int cur0 = st->cur0;
  const int cur = job == 0 ? cur0 : st->cur1[job - 1];
  const double* Sj = master + (size_t)(cur * (1 + k) + job) * mat;   // the job's own slot
  double* out = master + (size_t)((cur ^ 1) * (1 + k) + job) * mat;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ry = (lane >> 2) * RA, cx = (lane & 3) * CB;

  // epilogue elements of this thread: tid + 128 v, row-major in the tile
  double old[NE];
#pragma unroll
  for (int v = 0; v < NE; ++v) {
    const int e = tid + NT * v;
    const int64_t r = I * T + e / T, c = J * T + e % T;
    old[v] = (e < T * T && r < n && c < n) ? Sj[(size_t)r * Np + c] : 0.0;
  }

  double acc[RA][CB];
#pragma unroll
  for (int i = 0; i < RA; ++i)
#pragma unroll
    for (int j = 0; j < CB; ++j) acc[i][j] = 0.0;

  const int k1 = st->order >= 2 ? st->k1 : k;   // first-order directions
  const int passes = simt_job_passes(job, k1);
  const int nkb = (int)((n + BK - 1) / BK);     // K blocks per pass
  const int steps = passes * nkb;
  // The masters are exactly symmetric, so the K x T slab A[I rows][kb ..] is
  // read as rows kb .. kb + BK - 1, columns I T .. I T + T - 1 (contiguous)
  const double* A = nullptr;
  const double* B = nullptr;
  int lpass = 0, lkb = 0;   // position of the next load
  auto load = [&](int stage) {
    if (lkb == 0) {
      int mA, mB;
      simt_job_operands(job, lpass, k1, &mA, &mB);
      A = master + (size_t)((mA == 0 ? cur0 : st->cur1[mA - 1]) * (1 + k) + mA) * mat + I * T;
      B = master + (size_t)((mB == 0 ? cur0 : st->cur1[mB - 1]) * (1 + k) + mB) * mat + J * T;
    }
    double* s0 = sm + stage * 2 * SLAB;
#pragma unroll
    for (int v = 0; v < NCP; ++v) {
      const int idx = tid + NT * v;
      const int half = idx / (BK * T / 2), rem = idx % (BK * T / 2);
      const int row = rem / (T / 2), cq = 2 * (rem % (T / 2));
      const int64_t kr = (int64_t)lkb * BK + row;
      const double* g = (half ? B : A) + (size_t)(kr < n ? kr : 0) * Np + cq;
      cp_async16_zfill(s0 + half * SLAB + row * LD + cq, g, kr < n);
    }
    if (++lkb == nkb) {
      lkb = 0;
      ++lpass;
    }
  };
#pragma unroll
  for (int s = 0; s < STAGES - 1; ++s) {
    if (s < steps) load(s);
    cp_async_commit();
  }
  int stage = 0;
  for (int it = 0; it < steps; ++it) {
    cp_async_wait<STAGES - 2>();   // stage `it` has landed (this thread's copies)
    __syncthreads();               // ... and every thread's; stage it - 1 is free
    if (it + STAGES - 1 < steps) load(stage == 0 ? STAGES - 1 : stage - 1);
    cp_async_commit();
    const double* as = sm + stage * 2 * SLAB;
    const double* bs = as + SLAB;
#pragma unroll
    for (int q = 0; q < BK / 4; ++q) {
      const int kk = 4 * q + warp;
      double a[RA], b[CB];
#pragma unroll
      for (int i = 0; i < RA; ++i) a[i] = as[kk * LD + ry + i];
#pragma unroll
      for (int j = 0; j < CB; ++j) b[j] = bs[kk * LD + cx + j];
#pragma unroll
      for (int i = 0; i < RA; ++i)
#pragma unroll
        for (int j = 0; j < CB; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    if (++stage == STAGES) stage = 0;
  }
  cp_async_wait<0>();
  __syncthreads();

  // ---- fused epilogue
#pragma unroll
  for (int i = 0; i < RA; ++i)
#pragma unroll
    for (int j = 0; j < CB; ++j) sm[warp * T * T + (ry + i) * T + cx + j] = acc[i][j];
  __syncthreads();
  const double sg = (double)st->sigma_cur, om = 1.0 - sg;
  const bool write = job == 0 ? st->plan_write0 != 0 : true;
  double fnew = 0.0, fdiff = 0.0, tr = 0.0;
  double nw[NE];
  int bad = 0;
#pragma unroll
  for (int v = 0; v < NE; ++v) {
    const int e = tid + NT * v;
    nw[v] = 0.0;
    if (e >= T * T) continue;
    const int64_t r = I * T + e / T, c = J * T + e % T;
    if (r > c || c >= n) continue;   // owned by the mirrored element; outside (r <= c < n)
    const double x = (sm[e] + sm[T * T + e]) + (sm[2 * T * T + e] + sm[3 * T * T + e]);
    bad += isfinite(x) ? 0 : 1;
    const double y = sg * x + om * old[v];
    const double dd = old[v] - x;
    // elements off the diagonal count twice (a tile off the diagonal: below)
    fdiff = fma(diag && r != c ? 2.0 * dd : dd, dd, fdiff);
    if (write) {
      nw[v] = y;
      fnew = fma(diag && r != c ? 2.0 * y : y, y, fnew);
      if (r == c) tr += y;
      out[(size_t)r * Np + c] = y;
    }
  }
  red[0][tid] = fnew;
  red[1][tid] = fdiff;
  if (diag) {
    // diagonal elements lie T + 1 apart; a thread holds at most one of each
    // 32 consecutive ones
    if (tid < 32) red_tr[tid] = 0.0;
  }
  const int nbad = __syncthreads_count(bad);   // also: every sum has been read
  if (write) {
    constexpr int TS = T + 1;
#pragma unroll
    for (int v = 0; v < NE; ++v) {
      const int e = tid + NT * v;
      if (e < T * T) sm[(e / T) * TS + e % T] = nw[v];
      if (diag && e < T * T && e / T == e % T) red_tr[e / T] = tr;
    }
  }
  __syncthreads();
  if (write) {
    constexpr int TS = T + 1;
#pragma unroll
    for (int v = 0; v < NE; ++v) {   // the mirror (c, r), row-major in the mirror tile
      const int e = tid + NT * v;
      const int64_t c = J * T + e / T, r = I * T + e % T;
      if (e < T * T && r < c && c < n) out[(size_t)c * Np + r] = sm[(e % T) * TS + e / T];
    }
  }
  if (warp < 3) {
    double x = 0.0;
    if (warp < 2) {
      const double* p = red[warp];
      x = (p[lane] + p[lane + 32]) + (p[lane + 64] + p[lane + 96]);
    } else if (diag && write) {
      x = red_tr[lane];
    }
    if (warp < 2 || diag) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    }
    if (lane == 0) {
      double* p = partials + ((size_t)job * ptiles + blockIdx.x) * kNQ;
      if (warp == 0) {
        p[kQFroNew] = diag ? x : 2.0 * x;
        p[kQBad] = (double)nbad;
      } else if (warp == 1) {
        p[kQFroDiff] = diag ? x : 2.0 * x;
      } else {
        p[kQTrace] = x;
      }
    }
  }
}

// Tile edge of the FP32 form: 64 while the 128-wide tiles of every job would
// keep less than two thirds of the SMs busy; a 64-wide tile reads twice the
// shared memory per product.  Solve per layer, 128 / 64 wide: n = 700 k = 3 (84
// tiles) 145 / 101 us, n = 1000 k = 1 (72) 195 / 101 us, n = 1400 k = 1 (132)
// 267 / 280 us, n = 1000 k = 3 (144) 200 / 210 us, n = 4096 k = 1 3.53 / 4.43 ms.
inline int fp32_tile(int64_t n, int k) {
  const int64_t t = (n + 127) / 128;
  return t * (t + 1) / 2 * (1 + k) <= 100 ? 64 : 128;
}

// Per-device one-time setup: the SIMT layer kernels' dynamic shared memory
// exceeds the default 48 KB limit; thread-safe.
static void simt_setup() {
  constexpr int kDevices = 64;
  static std::once_flag once[kDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) return;
  std::call_once(once[dev], [] {
    cudaFuncSetAttribute(layer_simt_kernel<8, 16>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                         simt_smem_bytes<8, 16>());
    cudaFuncSetAttribute(layer_simt_kernel<4, 16>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                         simt_smem_bytes<4, 16>());
  });
}

cudaError_t launch_layer_simt(const Layout& L, void* ws, cudaStream_t s, int64_t* entries,
                              double* pass_flops) {
  char* base = (char*)ws;
  State* st = (State*)(base + L.off_state);
  double* partials = (double*)(base + L.off_partials);
  int64_t tiles = 0;
  if (L.precision == DMPT_FP64) {
    double* master = (double*)(base + L.off_master);
    const int bt = fp64_tile(L.n);
    tiles = fp64_tiles(L.n);
    const dim3 grid((unsigned)tiles, 1 + L.k);
    const auto kern = bt == 8 ? layer_fp64_kernel<8>
                              : (bt == 16 ? layer_fp64_kernel<16> : layer_fp64_kernel<32>);
    const cudaError_t e = launch_pdl(kern, grid, dim3(128), 0, s, st, master, L.n, L.Np, L.k,
                                     partials, L.partial_tiles);
    if (e != cudaSuccess) return e;
    if (pass_flops) *pass_flops = (double)tiles * bt * bt * (double)L.n * 2.0;
  } else {
    constexpr int smem8 = simt_smem_bytes<8, 16>(), smem4 = simt_smem_bytes<4, 16>();
    static_assert(2 * smem8 <= 227 * 1024 && 4 * smem4 <= 227 * 1024, "blocks per SM");
    simt_setup();
    const int bt = fp32_tile(L.n, L.k);
    const int64_t tb = (L.n + bt - 1) / bt;
    tiles = tb * (tb + 1) / 2;
    const cudaError_t e = launch_pdl(
        bt == 128 ? layer_simt_kernel<8, 16> : layer_simt_kernel<4, 16>,
        dim3((unsigned)tiles, 1 + L.k), dim3(256), bt == 128 ? smem8 : smem4, s, st,
        (float*)(base + L.off_master), L.n, L.Np, L.k, partials, L.partial_tiles);
    if (e != cudaSuccess) return e;
    if (pass_flops) *pass_flops = (double)tiles * bt * bt * (double)((L.n + 15) / 16 * 16) * 2.0;
  }
  if (entries) *entries = tiles;
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Dual split of the initial layer (Sec. II C, Eq. (DualMat2)):
//   hi = R16[2^e X],  lo = R16[2^e X - hi]   (round to nearest even),
// with e = s0_exp for S0 and s1_exp_cur[k] for S1_k (exact power-of-two
// scaling keeps FP16 values in range; BF16 uses e = 0).

template <typename H16>
__device__ __forceinline__ H16 to16(float x);
template <>
__device__ __forceinline__ __half to16<__half>(float x) { return __float2half_rn(x); }
template <>
__device__ __forceinline__ __nv_bfloat16 to16<__nv_bfloat16>(float x) {
  return __float2bfloat16_rn(x);
}
__device__ __forceinline__ float from16(__half x) { return __half2float(x); }
__device__ __forceinline__ float from16(__nv_bfloat16 x) { return __bfloat162float(x); }

__device__ __forceinline__ unsigned short bits16(__half x) { return __half_as_ushort(x); }
__device__ __forceinline__ unsigned short bits16(__nv_bfloat16 x) {
  return __bfloat16_as_ushort(x);
}

// Elements idx .. idx + 3 (idx a multiple of 4) of a master: x = src 2^e,
// hi = x rounded to 16 bits, lo = (x - hi) rounded to 16 bits.
template <typename H16>
__device__ __forceinline__ void split4(const float* __restrict__ src, unsigned short* hi,
                                       unsigned short* lo, size_t idx, int e) {
  const float4 v = __ldcg(reinterpret_cast<const float4*>(src + idx));
  const float x[4] = {ldexpf(v.x, e), ldexpf(v.y, e), ldexpf(v.z, e), ldexpf(v.w, e)};
  unsigned short hb[4], lb[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const H16 h = to16<H16>(x[t]);
    hb[t] = bits16(h);
    lb[t] = bits16(to16<H16>(x[t] - from16(h)));
  }
  *reinterpret_cast<uint2*>(hi + idx) =
      make_uint2(hb[0] | ((unsigned)hb[1] << 16), hb[2] | ((unsigned)hb[3] << 16));
  *reinterpret_cast<uint2*>(lo + idx) =
      make_uint2(lb[0] | ((unsigned)lb[1] << 16), lb[2] | ((unsigned)lb[3] << 16));
}

template <typename H16>
__global__ void split_kernel(const State* st, const float* __restrict__ master,
                             unsigned short* ops, int64_t Np, int k, int first_job) {
  pdl_wait();
  pdl_launch();
  const size_t mat = (size_t)Np * Np;   // a multiple of 4
  const int m = first_job + blockIdx.y;  // matrix: 0 = S0, 1 + j = S1_j
  const int cur = m == 0 ? st->cur0 : st->cur1[m - 1];
  const int e = m == 0 ? st->s0_exp : st->s1_exp_cur[m - 1];
  const float* src = master + (size_t)(cur * (1 + k) + m) * mat;
  const int zh = m == 0 ? st->z0_cur : zslice(cur, m, 0, k);
  unsigned short* hi = ops + (size_t)zh * mat;
  unsigned short* lo = ops + (size_t)(zh + 1) * mat;
  for (size_t i = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) * 4; i < mat;
       i += (size_t)gridDim.x * blockDim.x * 4)
    split4<H16>(src, hi, lo, i, e);
}

cudaError_t launch_split(const Layout& L, void* ws, int first_job, cudaStream_t s, int jobs) {
  char* base = (char*)ws;
  const State* st = (const State*)(base + L.off_state);
  const int64_t bx = L.Np * L.Np / 1024;   // 4 elements per thread
  const dim3 grid((unsigned)(bx < 152 * 4 ? bx : 152 * 4), jobs < 0 ? 1 + L.k - first_job : jobs);
  return launch_pdl(L.precision == DMPT_DUAL_FP16 ? split_kernel<__half>
                                                  : split_kernel<__nv_bfloat16>,
                    grid, dim3(256), 0, s, st, (const float*)(base + L.off_master),
                    (unsigned short*)(base + L.off_ops16), L.Np, L.k, first_job);
}

// ---------------------------------------------------------------------------
// Whole-matrix readers of the masters.  The tensor-core layer epilogue keeps
// an FP32 master in one orientation only (element (r, c) at (max, min): the
// lower triangle with the diagonal); the other kernels write both.  So a
// reader takes output tile (bi, bj) (kSymTile x kSymTile, 256 threads) from
// the lower tile (max(bi, bj), min(bi, bj)): loaded row by row (coalesced,
// every load of the tile in flight at once) into shared memory, written row
// by row, transposed where the output tile lies above the diagonal.
// `put(r, c, v)` writes the value of element (r, c), r, c < n.
constexpr int kSymTile = 64;
template <typename T, class Put>
__device__ __forceinline__ void sym_tile(const T* __restrict__ src, int64_t Np, int64_t n,
                                         int64_t bi, int64_t bj, T (*t)[kSymTile + 1], Put put) {
  constexpr int TS = kSymTile, RS = 256 / TS, RPT = TS / RS;   // 64 x 4 threads, 16 rows each
  const int tx = threadIdx.x % TS, ty = threadIdx.x / TS;
  const int64_t lr = TS * (bi > bj ? bi : bj), lc = TS * (bi > bj ? bj : bi);
  T v[RPT];
#pragma unroll
  for (int j = 0; j < RPT; ++j) v[j] = __ldcg(&src[(lr + ty + RS * j) * Np + lc + tx]);
#pragma unroll
  for (int j = 0; j < RPT; ++j) t[ty + RS * j][tx] = v[j];
  __syncthreads();
#pragma unroll
  for (int j = 0; j < RPT; ++j) {
    const int i = ty + RS * j;
    const int64_t r = TS * bi + i, c = TS * bj + tx;
    if (r < n && c < n) {
      const T x = bi > bj ? t[i][tx] : (bi < bj ? t[tx][i] : (tx <= i ? t[i][tx] : t[tx][i]));
      put(r, c, x);
    }
  }
  __syncthreads();   // the block's next tile reuses t
}

// ---------------------------------------------------------------------------
// Checkpoints of the S0 recursion (ckpt_every = k >= 2) and the recompute of a
// segment of states from its checkpoint in the backward pass.

__global__ void ckpt_store_kernel(const State* st, const float4* master,
                                  float4* ckpt, int64_t Np, int lk) {
  pdl_wait();
  pdl_launch();
  if (!st->ckpt_pending) return;
  const int slot = st->d0_updates / st->ckpt_k;
  if (slot >= st->ckpt_slots) return;   // cannot happen: slots cover max_layers / k + 1
  const size_t n4 = (size_t)Np * Np / 4;
  const float4* src = master + (size_t)st->cur0 * (1 + lk) * n4;
  float4* dst = ckpt + (size_t)slot * n4;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4;
       i += (size_t)gridDim.x * blockDim.x)
    dst[i] = __ldcg(&src[i]);
}

cudaError_t launch_ckpt_store(const Layout& L, void* ws, cudaStream_t s) {
  char* base = (char*)ws;
  return launch_pdl(ckpt_store_kernel, dim3(152 * 4), dim3(256), 0, s,
                    (const State*)(base + L.off_state), (const float4*)(base + L.off_master),
                    (float4*)(base + L.off_ckpt), L.Np, L.k);
}

// Checkpoint c (state a) into S0 master buffer 0; it becomes the current S0
// and its 16-bit copies go to the first tape slot (split afterwards).
__global__ void seg_load_kernel(State* st, float4* master, const float4* __restrict__ ckpt,
                                int64_t Np, int c, int a) {
  const size_t n4 = (size_t)Np * Np / 4;
  const float4* src = ckpt + (size_t)c * n4;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4;
       i += (size_t)gridDim.x * blockDim.x)
    master[i] = src[i];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st->cur0 = 0;
    st->z0_cur = st->tape_base;
    st->adj_seg_a = a;
  }
}

// The upper triangle of an Np x Np master from its lower triangle (a
// checkpoint of a state that a tensor-core layer wrote holds only the lower
// one; the hi/lo split that follows a reload reads the whole matrix).
__global__ void __launch_bounds__(256) mirror_lower_kernel(float* M, int64_t Np) {
  __shared__ float t[kSymTile][kSymTile + 1];
  const int64_t tb = Np / kSymTile;
  for (int64_t tile = blockIdx.x; tile < tb * tb; tile += gridDim.x) {
    const int64_t bi = tile / tb, bj = tile % tb;
    if (bi > bj) continue;   // uniform across the block: lower tiles are only read
    sym_tile<float>(M, Np, Np, bi, bj, t, [&](int64_t r, int64_t c, float v) { M[r * Np + c] = v; });
  }
}

// M[r][c] = M[c][r] for r > c, count matrices: lower output tile (bi, bj)
// from upper tile (bj, bi), loaded row by row and transposed through shared
// memory; a diagonal tile mirrors its own upper half.
__global__ void __launch_bounds__(256) mirror_upper_kernel(double* M, int64_t n, int64_t ld) {
  constexpr int TS = kSymTile, RS = 256 / TS, RPT = TS / RS;
  __shared__ double t[TS][TS + 1];
  double* A = M + (size_t)blockIdx.y * n * ld;
  const int tx = threadIdx.x % TS, ty = threadIdx.x / TS;
  const int64_t tb = (n + TS - 1) / TS;
  for (int64_t tile = blockIdx.x; tile < tb * tb; tile += gridDim.x) {
    const int64_t bi = tile / tb, bj = tile % tb;
    if (bi < bj) continue;   // uniform across the block: upper tiles are only read
    double v[RPT];
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      const int64_t r = TS * bj + ty + RS * j, c = TS * bi + tx;   // upper tile (bj, bi)
      v[j] = (r < n && c < n) ? A[r * ld + c] : 0.0;
    }
#pragma unroll
    for (int j = 0; j < RPT; ++j) t[ty + RS * j][tx] = v[j];
    __syncthreads();
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      const int i = ty + RS * j;
      const int64_t r = TS * bi + i, c = TS * bj + tx;
      if (r < n && c < n && r > c) A[r * ld + c] = t[tx][i];
    }
    __syncthreads();
  }
}

cudaError_t launch_mirror_upper(double* M, int64_t n, int64_t ld, int count, cudaStream_t s) {
  if (count < 1 || n < 1) return cudaSuccess;
  mirror_upper_kernel<<<dim3(152 * 8, count), 256, 0, s>>>(M, n, ld);
  return cudaGetLastError();
}

cudaError_t launch_seg_load(const Layout& L, void* ws, int c, int a, cudaStream_t s) {
  if (c < 0 || c >= L.ckpt_slots) return cudaErrorInvalidValue;
  char* base = (char*)ws;
  seg_load_kernel<<<152 * 4, 256, 0, s>>>((State*)(base + L.off_state),
                                          (float4*)(base + L.off_master),
                                          (const float4*)(base + L.off_ckpt), L.Np, c, a);
  mirror_lower_kernel<<<152 * 16, 256, 0, s>>>((float*)(base + L.off_master), L.Np);
  return cudaGetLastError();
}

// Plan the recompute of S_m = sigma_m S_{m-1}^2 + (1 - sigma_m) S_{m-1}: the
// square job only, S0 update stored, 16-bit copies into tape slot m - a.
__global__ void recompute_step_kernel(State* st, int after, int m, int a, int64_t item_base) {
  pdl_wait();
  if (m > 0) pdl_launch();   // the next kernel is a layer product, which reads after its wait
  st->round_ctr = 0u;
  if (after) {   // the layer's new state is the current S0
    st->cur0 ^= 1;
    st->z0_cur = st->z0_next;
    if (st->timeout_flag) {
      st->status = DMPT_ETIMEOUT;
      st->done = 1;
    }
  }
  st->item_base = m > 0 ? item_base : 0;
  st->plan_square = m > 0;
  st->plan_write0 = m > 0;
  if (m > 0) {
    st->sigma_cur = st->sigma[m];
    for (int j = 0; j < kMaxK; ++j) st->plan_resp[j] = 0;
    st->z0_next = st->tape_base + 2 * (m - a);
  }
}

cudaError_t launch_recompute_step(const Layout& L, void* ws, bool after, int m, int a,
                                  int64_t item_base, cudaStream_t s) {
  return launch_pdl(recompute_step_kernel, dim3(1), dim3(1), 0, s,
                    (State*)((char*)ws + L.off_state), (int)after, m, a, item_base);
}

// ---------------------------------------------------------------------------
// Adjoint of the S0 recursion (backward pass of L = Tr[G P]).
//   Gbar = (G + G^T) / 2 into response slot 1, buffer 0 (FP32 master), with
//   ||Gbar||_F^2 partial sums; and at the end dL/dH = -Gbar / (eps_N - eps_1)
//   (S0 = (eps_N I - H) / (eps_N - eps_1), bounds held fixed).

__global__ void __launch_bounds__(256) adj_init_kernel(const double* __restrict__ G, float* master,
                                                       int64_t n, int64_t Np, int64_t ld, int lk,
                                                       double* partials, int64_t ptiles) {
  // 32 x 32 tile pairs (bi <= bj): the upper tile in registers, the lower one
  // through shared memory; the mirror tile is the upper one's result transposed.
  // Two FP64 operations per element of the upper tile (the FP64 rate of the part
  // is low): the sum and the squared norm, which keeps FP64's range (G may be
  // tiny or huge).  n = 4096: 245 -> 79 us.
  __shared__ double dn[32][33];
  __shared__ float sv[32][33];
  __shared__ double red[2 * 256];
  const size_t mat = (size_t)Np * Np;
  float* dst = master + (size_t)1 * mat;   // buffer 0, slot 1
  (void)lk;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t TB = Np / 32;
  const int64_t pairs = TB * (TB + 1) / 2;
  double f = 0.0;
  int nbad = 0;
  for (int64_t tp = blockIdx.x; tp < pairs; tp += gridDim.x) {
    int64_t bj = (int64_t)((sqrtf(8.0f * (float)tp + 1.0f) - 1.0f) * 0.5f);
    while ((bj + 1) * (bj + 2) / 2 <= tp) ++bj;
    while (bj * (bj + 1) / 2 > tp) --bj;
    const int64_t bi = tp - bj * (bj + 1) / 2;
    double up[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int rl = ty + 8 * i;
      const int64_t r = bi * 32 + rl, c = bj * 32 + tx;
      const int64_t r2 = bj * 32 + rl, c2 = bi * 32 + tx;
      up[i] = (r < n && c < n) ? G[r * ld + c] : 0.0;
      dn[rl][tx] = (r2 < n && c2 < n) ? G[r2 * ld + c2] : 0.0;
    }
    __syncthreads();
    double ft = 0.0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int rl = ty + 8 * i;
      // (G + G^T)/2 at (r, c): up and the transposed element dn[tx][rl]
      const float v = narrow<1>(up[i] + dn[tx][rl]);
      dst[(size_t)(bi * 32 + rl) * Np + bj * 32 + tx] = v;
      sv[rl][tx] = v;
      const double w = widen(v);
      ft = fma(w, w, ft);
      nbad += isfinite(v) ? 0 : 1;
    }
    f += bi < bj ? 2.0 * ft : ft;
    __syncthreads();
    if (bi < bj) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int rl = ty + 8 * i;
        dst[(size_t)(bj * 32 + rl) * Np + bi * 32 + tx] = sv[tx][rl];
      }
    }
  }
  double v[2] = {f, (double)nbad};
  block_sum<2, 256>(v, red);
  if (threadIdx.x == 0) {
    double* p = partials + ((size_t)1 * ptiles + blockIdx.x) * kNQ;
    p[kQTrace] = 0.0;
    p[kQFroNew] = v[0];
    p[kQFroDiff] = 0.0;
    p[kQBad] = v[1];
  }
}

cudaError_t launch_adj_init(const Layout& L, void* ws, const double* G, int64_t ld, int blocks,
                            cudaStream_t s) {
  char* base = (char*)ws;
  adj_init_kernel<<<blocks, 256, 0, s>>>(G, (float*)(base + L.off_master), L.n, L.Np, ld, L.k,
                                         (double*)(base + L.off_partials), L.partial_tiles);
  return cudaGetLastError();
}

__global__ void __launch_bounds__(256) adj_finalize_kernel(const State* st,
                                                           const float* __restrict__ master,
                                                           double* dLdH, int64_t n, int64_t Np,
                                                           int64_t ld, int lk) {
  __shared__ float t[kSymTile][kSymTile + 1];
  const size_t mat = (size_t)Np * Np;
  const float* src = master + (size_t)(st->cur1[0] * (1 + lk) + 1) * mat;
  const double scale = -1.0 / (st->epsN - st->eps1);
  const int64_t tb = (n + kSymTile - 1) / kSymTile;
  for (int64_t tile = blockIdx.x; tile < tb * tb; tile += gridDim.x)
    sym_tile<float>(src, Np, n, tile / tb, tile % tb, t, [&](int64_t r, int64_t c, float v) {
      dLdH[r * ld + c] = scale * widen(v);
    });
}

cudaError_t launch_adj_finalize(const Layout& L, void* ws, double* dLdH, int64_t ld,
                                cudaStream_t s) {
  char* base = (char*)ws;
  adj_finalize_kernel<<<152 * 16, 256, 0, s>>>((const State*)(base + L.off_state),
                                              (const float*)(base + L.off_master), dLdH, L.n,
                                              L.Np, ld, L.k);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Outputs: P = S0, P1_k = S1_k (orthogonal basis, Z = I), as float64.

// Output element (r, c) of matrix y (0 = P, 1 + j = P1_j) from master value v;
// the complement form (the recursion ran on I - P) gives P = I - S0,
// P_o = -S_o.
__device__ __forceinline__ double out_value(double v, int64_t r, int64_t c, int y, bool hole) {
  return !hole ? v : (y == 0 ? (r == c ? 1.0 : 0.0) - v : -v);
}
__device__ __forceinline__ double out_value(float v, int64_t r, int64_t c, int y, bool hole) {
  if (!hole) return widen(v);
  if (y == 0) return r == c ? 1.0 - (double)v : widen(0.0f - v);   // 0 - 0 = +0, as in FP64
  return widen(-v);
}

template <typename T>
__global__ void __launch_bounds__(256) finalize_kernel(const State* st,
                                                       const T* __restrict__ master, double* P,
                                                       double* P1, int64_t n, int64_t Np,
                                                       int64_t ld, int k, int slot0) {
  // k: layout slots; grid.y = 1 + the number of blocks written to P1, which
  // come from slots slot0, slot0 + 1, ...; kSymTile x kSymTile output tiles
  __shared__ T t[kSymTile][kSymTile + 1];
  const size_t mat = (size_t)Np * Np;
  const int y = blockIdx.y;
  pdl_wait();
  pdl_launch();
  if (y == 0 && P == nullptr) return;
  const int m = y == 0 ? 0 : slot0 + y - 1;
  const int cur = m == 0 ? st->cur0 : st->cur1[m - 1];
  const T* src = master + (size_t)(cur * (1 + k) + m) * mat;
  double* dst = y == 0 ? P : P1 + (size_t)(y - 1) * n * ld;
  const bool hole = st->hole != 0;
  const int64_t tb = (n + kSymTile - 1) / kSymTile;
  for (int64_t tile = blockIdx.x; tile < tb * tb; tile += gridDim.x)
    sym_tile<T>(src, Np, n, tile / tb, tile % tb, t, [&](int64_t r, int64_t c, T v) {
      dst[r * ld + c] = out_value(v, r, c, y, hole);
    });
}

cudaError_t launch_finalize(const Layout& L, void* ws, double* P, double* P1, int64_t ld,
                            int k_out, cudaStream_t s, int slot0) {
  char* base = (char*)ws;
  const State* st = (const State*)(base + L.off_state);
  const int64_t tb = (L.n + kSymTile - 1) / kSymTile;
  const dim3 grid((unsigned)(tb * tb < 152 * 16 ? tb * tb : 152 * 16), 1 + k_out);
  if (L.precision == DMPT_FP64)
    return launch_pdl(finalize_kernel<double>, grid, dim3(256), 0, s, st,
                      (const double*)(base + L.off_master), P, P1, L.n, L.Np, ld, L.k, slot0);
  return launch_pdl(finalize_kernel<float>, grid, dim3(256), 0, s, st,
                    (const float*)(base + L.off_master), P, P1, L.n, L.Np, ld, L.k, slot0);
}

// n_occ = 0 (full = 0) or n_occ = n (full = 1): P = 0 or I, P1 = 0.
__global__ void trivial_kernel(int64_t n, int k, int64_t ld, int full, double* P, double* P1) {
  const int m = blockIdx.y;
  if (m == 0 && P == nullptr) return;
  double* dst = m == 0 ? P : P1 + (size_t)(m - 1) * n * ld;
  const int64_t total = n * n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i / n, c = i - r * n;
    dst[r * ld + c] = (m == 0 && full && r == c) ? 1.0 : 0.0;
  }
}

cudaError_t launch_trivial(int64_t n, int k, int64_t ld, int full, double* P, double* P1,
                           cudaStream_t s) {
  dim3 grid(152, 1 + k);
  trivial_kernel<<<grid, 256, 0, s>>>(n, k, ld, full, P, P1);
  return cudaGetLastError();
}

}  // namespace dmpt

namespace dmpt {
// *flag = 1 when every instance's control block (at base + offs[i]) says done
__global__ void batch_all_done_kernel(const char* base, const long long* offs, int count,
                                      int* flag) {
  int all = 1;
  for (int i = threadIdx.x; i < count; i += blockDim.x) {
    const State* st = (const State*)(base + offs[i]);
    if (!st->done) all = 0;
  }
  all = __syncthreads_and(all);
  if (threadIdx.x == 0) *flag = all;
}

cudaError_t launch_batch_all_done(const void* base, const long long* offs, int count, int* flag,
                                  cudaStream_t s) {
  batch_all_done_kernel<<<1, 256, 0, s>>>((const char*)base, offs, count, flag);
  return cudaGetLastError();
}

// out[b] = the control block at base + offs[b] (one block per instance), so
// that the host reads every instance's state with one copy.
__global__ void gather_states_kernel(const char* base, const long long* offs, State* out) {
  static_assert(sizeof(State) % 4 == 0, "State copied as words");
  const unsigned* src = (const unsigned*)(base + offs[blockIdx.x]);
  unsigned* dst = (unsigned*)(out + blockIdx.x);
  for (int i = threadIdx.x; i < (int)(sizeof(State) / 4); i += blockDim.x) dst[i] = src[i];
}

cudaError_t launch_gather_states(const void* base, const long long* offs, int count, State* out,
                                 cudaStream_t s) {
  if (count < 1) return cudaSuccess;
  gather_states_kernel<<<count, 256, 0, s>>>((const char*)base, offs, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Batched set-up and outputs of the batch path (one launch per step for every
// instance; the values are those of the single-instance kernels above).

// The instance that owns unit u: the largest i with first[i] <= u
// (first[0] = 0 <= u < first[count]).
__device__ __forceinline__ int batch_find(const int64_t* __restrict__ first, int count,
                                          int64_t u) {
  int lo = 0, hi = count - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (first[mid] <= u)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

// One block per instance: a zeroed control block with its fields, the bounds
// keys, and zero partial sums for the initial layer's blocks that hold no
// tile pair.
__global__ void __launch_bounds__(256) batch_setup_kernel(const BatchInst* __restrict__ bi,
                                                          BatchCommon c) {
  const BatchInst& b = bi[blockIdx.x];
  static_assert(sizeof(State) % 4 == 0, "State zeroed as words");
  unsigned* w = reinterpret_cast<unsigned*>(b.st);
  for (int i = threadIdx.x; i < (int)(sizeof(State) / 4); i += blockDim.x) w[i] = 0u;
  const int64_t empty = (int64_t)(kInitBlocks - b.init_blocks) * kNQ;
  for (int j = 0; j <= b.k; ++j) {
    double* p = b.partials + ((size_t)j * b.ptiles + b.init_blocks) * kNQ;
    for (int64_t e = threadIdx.x; e < empty; e += blockDim.x) p[e] = 0.0;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    state_init_fields(b.st, b.k, c.max_layers, c.precision, b.n_occ, c.c_pt, c.c_d0, 0,
                      4 * (1 + b.layout_k), 0, b.layout_k, b.n, 1, 0, c.fo, b.hole);
    long long* key = reinterpret_cast<long long*>(&b.st->eps1);
    key[0] = dkey(INFINITY);
    key[1] = dkey(-INFINITY);
  }
}

// Gershgorin discs (as bounds_rows_kernel): one warp per kBatchRows rows of
// one instance, each row's radius summed in the same lane order.
__global__ void batch_bounds_rows_kernel(const BatchInst* __restrict__ bi,
                                         const int64_t* __restrict__ first, int count) {
  const int lane = threadIdx.x & 31;
  const int64_t u = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (u >= first[count]) return;   // uniform across the warp
  const int i = batch_find(first, count, u);
  const BatchInst& b = bi[i];
  const int64_t r0 = (u - first[i]) * kBatchRows;
  double lo = INFINITY, hi = -INFINITY;
  for (int64_t r = r0; r < r0 + kBatchRows && r < b.n; ++r) {
    const double* row = b.H + r * b.ld;
    double s = 0.0;
    for (int64_t j = lane; j < b.n; j += 32) s += fabs(row[j]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const double d = row[r];
    const double rad = s - fabs(d);
    lo = fmin(lo, d - rad);
    hi = fmax(hi, d + rad);
  }
  if (lane == 0) {
    long long* key = reinterpret_cast<long long*>(&b.st->eps1);
    atomicMin(&key[0], dkey(lo));
    atomicMax(&key[1], dkey(hi));
  }
}

__global__ void batch_bounds_fin_kernel(const BatchInst* __restrict__ bi, int count) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  long long* key = reinterpret_cast<long long*>(&bi[i].st->eps1);
  const double lo = dkey_inv(key[0]);
  const double hi = dkey_inv(key[1]);
  bi[i].st->eps1 = lo;
  bi[i].st->epsN = hi;
}

// Initial layer: unit u is virtual block u - first[i] of instance i's grid of
// kInitBlocks blocks.
template <typename T>
__global__ void __launch_bounds__(256) batch_init_kernel(const BatchInst* __restrict__ bi,
                                                         const int64_t* __restrict__ first,
                                                         int count) {
  const int64_t u = blockIdx.x;
  const int i = batch_find(first, count, u);
  const BatchInst& b = bi[i];
  init_body<T>(b.st, static_cast<T*>(b.master), b.H, b.H1, b.n, b.Np, b.ld, b.k, 0, b.k,
               nullptr, b.partials, b.ptiles, u - first[i], kInitBlocks);
}

__global__ void __launch_bounds__(kDecideThreads)
    batch_decide_init_kernel(const BatchInst* __restrict__ bi) {
  __shared__ DecideShared sh;
  const BatchInst& b = bi[blockIdx.x];
  decide_body<false>(b.st, b.partials, b.ptiles, kInitBlocks, 1 + b.k, kDecideInit, sh);
}

// 16-bit split of matrices 0 .. layout k (as split_kernel), kBatchChunk
// elements per block, four per thread and step.
template <typename H16>
__global__ void __launch_bounds__(256) batch_split_kernel(const BatchInst* __restrict__ bi,
                                                          const int64_t* __restrict__ first,
                                                          int count) {
  const int64_t u = blockIdx.x;
  const int i = batch_find(first, count, u);
  const BatchInst& b = bi[i];
  const State* st = b.st;
  const int lk = b.layout_k;
  const size_t mat = (size_t)b.Np * b.Np;   // a multiple of 4
  const int64_t cpm = (int64_t)((mat + kBatchChunk - 1) / kBatchChunk);
  const int64_t c = u - first[i];
  const int m = (int)(c / cpm);
  const size_t e0 = (size_t)(c - (int64_t)m * cpm) * kBatchChunk;
  const int cur = m == 0 ? st->cur0 : st->cur1[m - 1];
  const int e = m == 0 ? st->s0_exp : st->s1_exp_cur[m - 1];
  const float* src = static_cast<const float*>(b.master) + (size_t)(cur * (1 + lk) + m) * mat;
  const int zh = m == 0 ? st->z0_cur : zslice(cur, m, 0, lk);
  unsigned short* hi = b.ops + (size_t)zh * mat;
  unsigned short* lo = b.ops + (size_t)(zh + 1) * mat;
#pragma unroll
  for (int q = 0; q < kBatchChunk / (4 * 256); ++q) {
    const size_t idx = e0 + (size_t)(q * 256 + threadIdx.x) * 4;
    if (idx >= mat) break;
    split4<H16>(src, hi, lo, idx, e);
  }
}

// Outputs (as finalize_kernel with slot0 = 1): unit c of matrix y (0 = P,
// 1 + j = P1_j) is output tile c of that matrix (kSymTile x kSymTile tiles,
// row-major).
template <typename T>
__global__ void __launch_bounds__(256) batch_finalize_kernel(const BatchInst* __restrict__ bi,
                                                             const int64_t* __restrict__ first,
                                                             int count) {
  __shared__ T t[kSymTile][kSymTile + 1];
  const int64_t u = blockIdx.x;
  const int i = batch_find(first, count, u);
  const BatchInst& b = bi[i];
  const int64_t n = b.n;
  const int64_t tb = (n + kSymTile - 1) / kSymTile;
  const int64_t c = u - first[i];
  const int y = (int)(c / (tb * tb));
  if (y == 0 && b.P == nullptr) return;
  const int64_t tile = c - (int64_t)y * tb * tb;
  const State* st = b.st;
  const size_t mat = (size_t)b.Np * b.Np;
  const int cur = y == 0 ? st->cur0 : st->cur1[y - 1];
  const T* src = static_cast<const T*>(b.master) + (size_t)(cur * (1 + b.layout_k) + y) * mat;
  double* dst = y == 0 ? b.P : b.P1 + (size_t)(y - 1) * n * b.ld;
  const bool hole = st->hole != 0;
  const int64_t ld = b.ld;
  sym_tile<T>(src, b.Np, n, tile / tb, tile % tb, t, [&](int64_t r, int64_t cc, T v) {
    dst[r * ld + cc] = out_value(v, r, cc, y, hole);
  });
}

cudaError_t launch_batch_setup(const BatchInst* bi, const int64_t* first, int count,
                               const BatchCommon& c, const int64_t* units, bool dual, bool bf16,
                               cudaStream_t s) {
  if (count < 1) return cudaSuccess;
  const int64_t* f_rows = first + kBsRows * (count + 1);
  const int64_t* f_init = first + kBsInit * (count + 1);
  const int64_t* f_split = first + kBsSplit * (count + 1);
  batch_setup_kernel<<<count, 256, 0, s>>>(bi, c);
  batch_bounds_rows_kernel<<<(unsigned)((units[kBsRows] * 32 + 255) / 256), 256, 0, s>>>(
      bi, f_rows, count);
  batch_bounds_fin_kernel<<<(count + 255) / 256, 256, 0, s>>>(bi, count);
  if (c.precision == DMPT_FP64)
    batch_init_kernel<double><<<(unsigned)units[kBsInit], 256, 0, s>>>(bi, f_init, count);
  else
    batch_init_kernel<float><<<(unsigned)units[kBsInit], 256, 0, s>>>(bi, f_init, count);
  batch_decide_init_kernel<<<count, kDecideThreads, 0, s>>>(bi);
  if (dual && units[kBsSplit] > 0) {
    if (bf16)
      batch_split_kernel<__nv_bfloat16><<<(unsigned)units[kBsSplit], 256, 0, s>>>(bi, f_split,
                                                                                  count);
    else
      batch_split_kernel<__half><<<(unsigned)units[kBsSplit], 256, 0, s>>>(bi, f_split, count);
  }
  return cudaGetLastError();
}

cudaError_t launch_batch_finalize(const BatchInst* bi, const int64_t* first, int count,
                                  int64_t units, bool fp64, cudaStream_t s) {
  if (count < 1 || units < 1) return cudaSuccess;
  const int64_t* f_out = first + kBsOut * (count + 1);
  if (fp64)
    batch_finalize_kernel<double><<<(unsigned)units, 256, 0, s>>>(bi, f_out, count);
  else
    batch_finalize_kernel<float><<<(unsigned)units, 256, 0, s>>>(bi, f_out, count);
  return cudaGetLastError();
}
}  // namespace dmpt

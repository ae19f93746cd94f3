// ttsh_fno_fused.cuh - the corrector network's layers as two kernels each, forward and backward
// (included by ttsh_fno.cu; grids up to 512 x 512, an even number of at most 16 kept modes).
//
//   row kernel     one (sample, y) grid row at a time: the inverse row transform of the spectral
//                  part and the channel mixing as tensor-core products into two tensor-memory
//                  accumulators, their sum, bias and activation in registers, and the row
//                  transform of the result onto the kept kx straight from shared memory.  A
//                  layer's activations cross memory once in each direction.
//   column kernel  one (kx, sample) per cluster of CS blocks: the transform along y onto the kept
//                  ky, the per-mode complex mixing and the inverse transform along y, the mixed
//                  modes exchanged through distributed shared memory.
//
// Spectral columns on their way to the column kernel lie as [b][kx][y][channel] (Re, Im) pairs,
// so that a block's column is one contiguous piece; on their way back as [b][k][y][channel]
// (k = Re kx 0..m-1, then Im), the order of the expanding products' K.  Every FP32 sum runs in the order of the separate kernels these
// replace, so that results, including every rounding to BF16, are the same bits.
#pragma once

#include <type_traits>

namespace fno_dev {

__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// One warp waits for the kernel ahead, the others at the block barrier: threads in
// griddepcontrol.wait take issue slots from the kernel they wait for.
__device__ __forceinline__ void pdl_wait_block() {
  if (threadIdx.x < 32) asm volatile("griddepcontrol.wait;" ::: "memory");
  __syncthreads();
}
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_all;\n" ::: "memory");
}

// ---------------------------------------------------------------------------------------
// Row kernel
//
// Bound at batch 8 by memory in the backward pass (217 MB, 32 us at the measured copy rate; 35-42 us)
// and by erf and exp besides in the forward one (218 MB with what the backward pass needs; 55-64
// us); at batch 1 by its chain of phases (8 us, of which 0.6 us wait for the columns, 0.5 us the
// products, 2 us the activation, 1.5 us the contraction).  The launches it replaces (expand,
// channel mixing, contract) took 38 us at batch 1 and 134 us (forward, training) at batch 8.
// One thread holds the 32 channels of one point, so that activation and projection need no
// exchange; the A tile of the next row travels while a block works on this one.
// ---------------------------------------------------------------------------------------
enum RowMode {
  R_LIFT = 0,        // h_0 = x Wp + bp, contracted with Fx
  R_FWD = 1,         // z = h W + b + s; h' = GELU(z), contracted with Fx
  R_LAST = 2,        // z = h W + b + s; y = z Wq + bq
  R_LAST_TRAIN = 3,  // the same, then the loss, dz = dy Wq, contracted with Bx^T
  R_BWD = 4,         // dh = dz W^T + adjoint spectral part; dz' = dh GELU'(z'), contracted with Bx^T
  R_BWD_FIRST = 5    // dh = dz W^T + adjoint spectral part
};

struct RowArgs {
  const __nv_bfloat16* A;    // [P][32]: h_l (forward) or dz_l (backward)
  const __nv_bfloat16* W;    // 32 x 32, [o][i]
  const __nv_bfloat16* E;    // [n][32]: matrix that expands the kept kx to the row
  const float* Z;            // [B][J][n][32]: columns to expand
  const __nv_bfloat16* C;    // [32][n]: matrix that contracts the row to the kept kx, rows Re 0, Im 0, Re 1, ...
  float2* X;                 // [B][m][n][32]: contracted columns
  const float* bias;         // 32
  const float* x;            // R_LIFT: [P][4], the caller's
  int x16;                   // 1: x is 16-byte aligned
  const float *Wp, *bp;      // R_LIFT
  const float* gin;          // R_BWD: GELU'(z) of the layer below
  float* gout;               // R_FWD in training: GELU'(z); R_LAST_TRAIN: z
  float* hout;               // R_FWD in training: GELU(z)
  __nv_bfloat16* hb;         // result in BF16: h_{l+1}, or dz
  float* dz;                 // R_BWD: dz', R_BWD_FIRST: dh
  const float *Wq, *bq;      // R_LAST*
  float* out;                // R_LAST*: [P]
  const float* target;       // R_LAST_TRAIN: [P]
  float* dout;               // R_LAST_TRAIN: [P]
  double* lpart;             // R_LAST_TRAIN: sum of squared errors of each grid row
  int n, J, tiles;           // tiles: A tiles in shared memory, 2 if some block has several rows
  long long Q, P;            // grid rows, points
  int* err;
};

__host__ __device__ constexpr bool row_has_mma(int mode) { return mode != R_LIFT; }
__host__ __device__ constexpr bool row_contracts(int mode) { return mode != R_LAST && mode != R_BWD_FIRST; }
__host__ __device__ constexpr bool row_stages(int mode, bool train) {   // FP32 rows through shared memory
  return mode == R_BWD || mode == R_BWD_FIRST || mode == R_LAST_TRAIN || (mode == R_FWD && train);
}

// Dynamic shared memory: A tile, `tiles` times (two where a block walks over several grid rows) |
// C | E | W | Z operand | FP32 rows of every warp, and 128 bytes to align the base.
inline int row_smem(int mode, bool train, int n, int tiles) {
  const int nr = n < 128 ? 128 : n;
  return 128 + tiles * nr * 64 + 64 * n + 2048 + (row_has_mma(mode) ? nr * 64 + 2048 : 0) +
         (row_stages(mode, train) ? nr * 128 : 0);
}

// 16-byte piece i of row r in a warp's 32 x 128-byte block, rotated so that both a thread's own
// row and a warp's consecutive pieces meet every bank once.
__device__ __forceinline__ float4* row_piece(unsigned char* blk, int r, int i) {
  return reinterpret_cast<float4*>(blk + r * 128 + ((i ^ (r & 7)) << 4));
}

// Blocks per SM the row kernel is compiled for (registers) and launched with where a block walks
// over several rows.
__host__ __device__ constexpr int row_blocks(int T, bool train) { return T == 4 ? 1 : (train ? 4 : 6) / T; }

template <int MODE, int T, bool TRAIN>
__global__ void __launch_bounds__(128 * T, row_blocks(T, TRAIN)) row_layer_kernel(RowArgs a) {
  constexpr int NT = 128 * T;
  // per x tile: 32 columns for the channel mixing, 32 for the expansion
  constexpr int TCOLS = row_has_mma(MODE) ? 64 * T : 32;
  extern __shared__ __align__(16) unsigned char row_dyn[];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_base;
  __shared__ float sc[CW * 6];    // bias / Wp, bp / Wq
  __shared__ double lred[4 * T];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = T == 1 ? a.n : 128 * T;   // T = 1 serves every grid up to 128
  constexpr int nr = 128 * T;
  const int J = a.J;
  unsigned char* base = row_dyn + ((128u - (smem_u32(row_dyn) & 127u)) & 127u);
  unsigned char* sA = base;
  unsigned char* sC = sA + a.tiles * nr * 64;
  unsigned char* sE = sC + 64 * n;
  unsigned char* sW = sE + (row_has_mma(MODE) ? nr * 64 : 0);
  unsigned char* sZ = sW + 2048;
  unsigned char* blk = sZ + (row_has_mma(MODE) ? 2048 : 0) + warp * 4096;

  // ---- operands that no kernel of this pass writes ----
  if constexpr (row_contracts(MODE)) {
    const int nk = n >> 3;
    for (int c = tid; c < 32 * nk; c += NT) {
      const int r = c / nk, kc = c % nk;
      cp_async16(sC + (r >> 3) * (n * 16) + kc * 128 + (r & 7) * 16, a.C + (long long)r * n + kc * 8);
    }
  }
  if constexpr (row_has_mma(MODE)) {
    for (int c = tid; c < n * 4; c += NT) cp_async16(sE + core_off(c >> 2, c & 3), a.E + c * 8);
    for (int c = tid; c < CW * 4; c += NT) cp_async16(sW + core_off(c >> 2, c & 3), a.W + c * 8);
  }
  // the first row's A tile: its writer finished before the kernel ahead of this one began
  long long q = blockIdx.x;
  if constexpr (row_has_mma(MODE)) {
    if (q < a.Q)
      for (int c = tid; c < n * 4; c += NT) cp_async16(sA + core_off(c >> 2, c & 3), a.A + q * n * CW + c * 8);
  }
  if constexpr (MODE == R_LIFT) {
    for (int c = tid; c < 5 * CW; c += NT) sc[c] = c < 4 * CW ? a.Wp[c] : a.bp[c - 4 * CW];
  } else if constexpr (MODE == R_FWD) {
    if (tid < CW) sc[tid] = a.bias[tid];
  } else if constexpr (MODE == R_LAST || MODE == R_LAST_TRAIN) {
    if (tid < CW) {
      sc[tid] = a.bias[tid];
      sc[CW + tid] = a.Wq[tid];
    }
    if (tid == CW) sc[2 * CW] = a.bq[0];
  }
  if (tid == 0) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar)) : "memory");
  if (warp == 0) tc_alloc(&tmem_base, TCOLS);
  const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
  const int tile = warp >> 2;
  const int x = tid;               // this thread's point of the grid row
  const bool live = x < n;
  const int wrows = n - warp * 32 >= 32 ? 32 : (n - warp * 32 > 0 ? n - warp * 32 : 0);
  uint32_t phase = 0;
  pdl_wait_block();
  if constexpr (!row_has_mma(MODE)) pdl_launch();

  // columns to expand: eight k of one channel a thread of the first four warps
  float zc[8];
  auto load_z = [&](long long qq) {
    const long long bb = qq / n, yy = qq - bb * n;
    const float* zp = a.Z + ((bb * J + warp * 8) * n + yy) * CW + lane;
#pragma unroll
    for (int i = 0; i < 8; ++i) zc[i] = warp * 8 + i < J ? zp[(long long)i * n * CW] : 0.f;
  };
  if constexpr (row_has_mma(MODE)) {
    if (warp < 4 && q < a.Q) load_z(q);
  }
  cp_async_wait();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  for (; q < a.Q; q += gridDim.x) {
    const long long p0 = q * n;
    const int b = (int)(q / n), y = (int)(q - (long long)b * n);
    uint32_t acc[CW];
    float v[CW];
    if constexpr (row_has_mma(MODE)) {
      if constexpr (MODE == R_BWD) {   // GELU' of the layer below, needed after the products
        for (int i = lane; i < wrows * 8; i += 32)
          cp_async16(row_piece(blk, i >> 3, i & 7), a.gin + (p0 + warp * 32) * CW + i * 4);
        asm volatile("cp.async.commit_group;" ::: "memory");
      }
      if (warp < 4) {   // K-major operand [channel][k]
        __nv_bfloat16 e[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) e[i] = __float2bfloat16_rn(zc[i]);
        *reinterpret_cast<uint4*>(sZ + core_off(lane, warp)) = *reinterpret_cast<const uint4*>(e);
      }
      asm volatile("cp.async.wait_group %0;" ::"n"(MODE == R_BWD ? 1 : 0) : "memory");   // this row's A tile
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> tensor core
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (tid == 0) {
        constexpr uint32_t id = umma_idesc_bf16(kTcRows, CW);
#pragma unroll
        for (int t = 0; t < T; ++t)
#pragma unroll
          for (int ks = 0; ks < 2; ++ks) {
            tc_mma_bf16(tmem + t * 64, umma_desc(smem_u32(sA) + t * 8192 + ks * 256, 128, 512),
                        umma_desc(smem_u32(sW) + ks * 256, 128, 512), id, ks);
            tc_mma_bf16(tmem + t * 64 + 32, umma_desc(smem_u32(sE) + t * 8192 + ks * 256, 128, 512),
                        umma_desc(smem_u32(sZ) + ks * 256, 128, 512), id, ks);
          }
        tc_commit(&mbar);
      }
      // the next row's inputs travel while this one is worked on
      const long long qn = q + gridDim.x;
      if (qn < a.Q) {
        unsigned char* nx = base + (sA == base ? nr * 64 : 0);
        for (int c = tid; c < n * 4; c += NT) cp_async16(nx + core_off(c >> 2, c & 3), a.A + qn * n * CW + c * 8);
        if (warp < 4) load_z(qn);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      const bool done = ttsh::mbar_wait_bounded(smem_u32(&mbar), phase, ttsh::kWaitLimitNs);
      if (__syncthreads_or(!done)) {
        if (tid == 0) atomicExch(a.err, 1);
        break;
      }
      phase ^= 1u;
      pdl_launch();   // the next kernel's blocks stage their operands under the epilogue
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      tc_ld32(tmem + lanes + tile * 64, acc);
#pragma unroll
      for (int c = 0; c < CW; ++c) v[c] = __uint_as_float(acc[c]);
      tc_ld32(tmem + lanes + tile * 64 + 32, acc);
#pragma unroll
      for (int c = 0; c < CW; ++c) {
        v[c] = v[c] + __uint_as_float(acc[c]);
        if constexpr (MODE == R_FWD || MODE == R_LAST || MODE == R_LAST_TRAIN) v[c] += sc[c];
      }
    } else {
      float4 xv = make_float4(0, 0, 0, 0);
      if (live) {
        const float* xp = a.x + (p0 + x) * 4;
        if (a.x16) xv = *reinterpret_cast<const float4*>(xp);
        else xv = make_float4(xp[0], xp[1], xp[2], xp[3]);
      }
#pragma unroll
      for (int c = 0; c < CW; ++c)
        v[c] = fmaf(xv.w, sc[3 * CW + c], fmaf(xv.z, sc[2 * CW + c], fmaf(xv.y, sc[CW + c], fmaf(xv.x, sc[c], sc[4 * CW + c]))));
    }

    // ---- FP32 rows that leave the kernel (or, R_BWD, that were staged) ----
    auto put_rows = [&]() {
#pragma unroll
      for (int i = 0; i < 8; ++i) *row_piece(blk, lane, i) = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    };
    auto store_rows = [&](float* dst) {
      __syncwarp();
      for (int i = lane; i < wrows * 8; i += 32)
        *reinterpret_cast<float4*>(dst + (p0 + warp * 32) * CW + i * 4) = *row_piece(blk, i >> 3, i & 7);
    };
    if constexpr (MODE == R_LAST_TRAIN) {
      put_rows();
      store_rows(a.gout);
    }
    if constexpr (MODE == R_FWD) {
      if constexpr (TRAIN) {   // GELU' for the backward pass, while erf(z / sqrt 2) is at hand
        float h[CW];
#pragma unroll
        for (int c = 0; c < CW; ++c) {
          h[c] = gelu(v[c]);
          v[c] = gelu_grad(v[c]);
        }
        put_rows();
        store_rows(a.gout);
#pragma unroll
        for (int c = 0; c < CW; ++c) v[c] = h[c];
        __syncwarp();
        put_rows();
        store_rows(a.hout);
      } else {
#pragma unroll
        for (int c = 0; c < CW; ++c) v[c] = gelu(v[c]);
      }
    }
    if constexpr (MODE == R_LAST || MODE == R_LAST_TRAIN) {
      float o = sc[2 * CW];
#pragma unroll
      for (int c = 0; c < CW; ++c) o = fmaf(v[c], sc[CW + c], o);
      if (live) a.out[p0 + x] = o;
      if constexpr (MODE == R_LAST_TRAIN) {
        double sq = 0.0;
        float g = 0.f;
        if (live) {
          const float r = o - a.target[p0 + x];
          sq = (double)r * r;
          g = 2.f * r / (float)a.P;
          a.dout[p0 + x] = g;
        }
#pragma unroll
        for (int c = 0; c < CW; ++c) v[c] = g * sc[CW + c];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) sq += __shfl_down_sync(0xffffffffu, sq, off);
        if (lane == 0) lred[warp] = sq;
      }
    }
    if constexpr (MODE == R_BWD) {
      asm volatile("cp.async.wait_group 1;" ::: "memory");   // all but the next row's tile
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 g = *row_piece(blk, lane, i);
        v[4 * i] *= g.x;
        v[4 * i + 1] *= g.y;
        v[4 * i + 2] *= g.z;
        v[4 * i + 3] *= g.w;
      }
    }
    if constexpr (MODE == R_BWD || MODE == R_BWD_FIRST) {
      put_rows();
      store_rows(a.dz);
      __syncwarp();   // read before the next row's copies
    }

    if constexpr (row_contracts(MODE)) {
      // The BF16 row as the tensor core's operand, in the layout the channel mixing reads it in
      // ([x][channel] core matrices): the contraction over x reads the same tile with the
      // channel as the M index (32 of 128 rows; the others are neighbouring points' values,
      // whose products nobody reads).
      if (live) {
#pragma unroll
        for (int kc = 0; kc < 4; ++kc) {
          __nv_bfloat162 e[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) e[i] = __floats2bfloat162_rn(v[kc * 8 + 2 * i], v[kc * 8 + 2 * i + 1]);
          *reinterpret_cast<uint4*>(sA + core_off(x, kc)) = *reinterpret_cast<const uint4*>(e);
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (tid == 0) {
        constexpr uint32_t id = umma_idesc_bf16(kTcRows, CW) | (1u << 15);   // A is MN-major
        for (int ks = 0; ks < n / 16; ++ks)
          tc_mma_bf16(tmem, umma_desc(smem_u32(sA) + ks * 1024, 512, 128),
                      umma_desc(smem_u32(sC) + ks * 256, 128, n * 16), id, ks);
        tc_commit(&mbar);
      }
      for (int c = tid; c < n * 4; c += NT)
        *reinterpret_cast<uint4*>(a.hb + p0 * CW + c * 8) = *reinterpret_cast<const uint4*>(sA + core_off(c >> 2, c & 3));
      if constexpr (MODE == R_LAST_TRAIN) {
        if (tid == 0) {
          double s = 0.0;
          for (int w = 0; w < 4 * T; ++w) s += lred[w];
          a.lpart[q] = s;
        }
      }
      const bool done = ttsh::mbar_wait_bounded(smem_u32(&mbar), phase, ttsh::kWaitLimitNs);
      if (__syncthreads_or(!done)) {
        if (tid == 0) atomicExch(a.err, 1);
        break;
      }
      phase ^= 1u;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (warp == 0) {   // accumulator rows 0..31: lane = channel, column = k
        tc_ld32(tmem, acc);
        float2* xo = a.X + ((long long)b * (J / 2) * n + y) * CW + lane;
#pragma unroll
        for (int k = 0; k < CW / 2; ++k)
          if (2 * k < J) xo[(long long)k * n * CW] = make_float2(__uint_as_float(acc[2 * k]), __uint_as_float(acc[2 * k + 1]));
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");   // accumulators read before reuse
    if constexpr (row_has_mma(MODE)) sA = base + (sA == base ? nr * 64 : 0);
  }
  cp_async_wait();   // a row left early (failed wait) may have copies in flight
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) tc_dealloc(tmem, TCOLS);
}

// ---------------------------------------------------------------------------------------
// Column kernel
// ---------------------------------------------------------------------------------------
struct ColArgs {
  const float2* X;                     // [B][m][n][32]
  const float2* G;                     // [J][n]: exp(-2 pi i ky y / n)
  const float *Gr, *Gi;                // the same, planar
  const __nv_bfloat16 *Wr, *Wi;        // [J][m][32][32]
  float *Hr, *Hi;                      // [B][J][m][32]: modes before the mixing (null: not kept)
  float* Z;                            // [B][J][n][32]
  int n, m;
  int ring;                            // pieces of X in shared memory at a time
  int* err;
};

// Forward (ADJ = false): H_j = sum_y G_jy X_y, Y = W H per mode, Z_y = sum_j conj(G_jy) Y_j.
// Adjoint: the same transforms around dH = W^H dY.  Block `rank` of the cluster transforms PB pairs
// of kept ky, mixes them, and afterwards transforms back n / CS values of y.
//
// Bound by what shared memory delivers to registers (4 bytes a lane and cycle, broadcast or not):
// a thread therefore sums ky and -ky of one channel together, whose G are each other's
// conjugates (ky = 0, whose G is 1, goes with -m), and transforms back four y of two channels.
// Measured at 256^2, 16 modes: the first sum 3.5 us with one ky a thread, 5.8 us with 8 ky in
// each of 4 blocks, 3.0 us so; the kernel 10 us at batch 1 and 33 us at batch 8 (268 MFLOP, 8 TFLOP/s;
// its 17 MB of columns would take 2.5 us), where the separate kernels took 23 and 57 us.
constexpr int kColThreads = 256;
constexpr int CS = 8;   // blocks per cluster
// BF16 values between the rows of a staged 32 x 32 weight: the adjoint reads a row per lane in
// 16-byte pieces, and 80 bytes apart eight of them meet every bank once.
__host__ __device__ constexpr int col_wrow(bool adj) { return adj ? 40 : CW; }
// X passes through a ring of pieces of 64 y (16 KB): all of them in shared memory where a block has
// an SM to itself anyway, two where further blocks then fit beside it.
__host__ __device__ constexpr int col_piece(int n) { return n < 64 ? n : 64; }
constexpr int kColRing = 8;

inline int col_smem(int n, int m, int ring, bool adj) {
  const int PB = (m + CS - 1) / CS, ny = n / CS < 4 ? 4 : n / CS;
  return 128 + ring * col_piece(n) * CW * 8 + PB * n * 8 + 4 * m * ny * 4 + 4 * PB * CW * col_wrow(adj) * 2 +
         2 * PB * CW * 8 + 2 * m * CW * 8;
}

template <bool ADJ>
__global__ void __launch_bounds__(kColThreads) column_layer_kernel(ColArgs a) {
  extern __shared__ __align__(16) unsigned char col_dyn[];
  __shared__ __align__(8) uint64_t mbar[kColRing];
  const int tid = threadIdx.x, warp = tid >> 5, c = tid & 31;
  const int n = a.n, m = a.m, J = 2 * m;
  const int kx = blockIdx.x / CS, rank = blockIdx.x % CS, b = blockIdx.y;
  const int PB = (m + CS - 1) / CS, t0 = rank * PB, tn = m - t0 < PB ? (m - t0 > 0 ? m - t0 : 0) : PB;
  const int ny = n / CS < 4 ? 4 : n / CS, y0 = rank * ny;   // this block's y (none where y0 >= n)
  // rows of the pair t: the one whose G is read, and its mirror image
  auto row_a = [m](int t) { return t == 0 ? m : t; };
  auto row_b = [m](int t) { return t == 0 ? 0 : 2 * m - t; };
  constexpr int WROW = col_wrow(ADJ), WMAT = CW * WROW;
  unsigned char* base = col_dyn + ((128u - (smem_u32(col_dyn) & 127u)) & 127u);
  const int piece = col_piece(n), pieces = n / piece, ring = a.ring;
  float2* xs = reinterpret_cast<float2*>(base);               // [ring][piece][32]
  float2* gs = xs + ring * piece * CW;                        // [PB][n]
  float* vr = reinterpret_cast<float*>(gs + PB * n);          // [J][ny]: this block's y of every ky row
  float* vi = vr + J * ny;
  float2* ys = reinterpret_cast<float2*>(vi + J * ny);        // [J][32]: every mixed mode
  float2* hs = ys + J * CW;                                   // [2 PB][32]: this block's modes
  __nv_bfloat16* wr = reinterpret_cast<__nv_bfloat16*>(hs + 2 * PB * CW);   // [2 PB][32][WROW]
  __nv_bfloat16* wi = wr + 2 * PB * WMAT;

  if (tid == 0) {
    for (int i = 0; i < ring; ++i)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar[i])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");   // this block has started
  const int lg = 31 - __clz(n / 2);   // n / 2 and ny / 4 are powers of two
  for (int e = tid; e < tn * (n / 2); e += kColThreads) {
    const int tl = e >> lg, r = e & ((1 << lg) - 1);
    cp_async16(gs + tl * n + 2 * r, a.G + (long long)row_a(t0 + tl) * n + 2 * r);
  }
  if (y0 < n) {
    const int lq = 31 - __clz(ny / 4);
    for (int e = tid; e < J * ny / 4; e += kColThreads) {
      const int j = e >> lq, r = e & ((1 << lq) - 1);
      cp_async16(vr + 4 * e, a.Gr + (long long)j * n + y0 + 4 * r);
      cp_async16(vi + 4 * e, a.Gi + (long long)j * n + y0 + 4 * r);
    }
  }
  for (int e = tid; e < 2 * tn * (CW * CW / 8); e += kColThreads) {
    const int jl = e / (CW * CW / 8), r = e % (CW * CW / 8), t = t0 + (jl >> 1);
    const long long src = ((long long)(jl & 1 ? row_b(t) : row_a(t)) * m + kx) * CW * CW + 8 * r;
    const int dst = jl * WMAT + (r >> 2) * WROW + 8 * (r & 3);
    cp_async16(wr + dst, a.Wr + src);
    cp_async16(wi + dst, a.Wi + src);
  }
  pdl_wait_block();   // (and the barriers are initialised)
  pdl_launch();
  auto load_piece = [&](int k) {   // thread 0: piece k of X into its place in the ring
    const uint32_t bytes = (uint32_t)(piece * CW * 8), bar = smem_u32(&mbar[k % ring]);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(xs + (k % ring) * piece * CW)), "l"(a.X + (((long long)b * m + kx) * n + k * piece) * CW),
                 "r"(bytes), "r"(bar) : "memory");
  };
  if (tid == 0)
    for (int k = 0; k < ring; ++k) load_piece(k);
  cp_async_wait();
  __syncthreads();

  // ---- H_j = sum over y, in order: a warp takes a pair of ky, a lane a channel; the next eight y
  // are loaded while these are summed (PB <= 2 pairs a block) ----
  {
    const bool on = warp < tn;
    float ar[2] = {0, 0}, ai[2] = {0, 0}, br[2] = {0, 0}, bi[2] = {0, 0};
    for (int k = 0; k < pieces; ++k) {
      if (!ttsh::mbar_wait_bounded(smem_u32(&mbar[k % ring]), (k / ring) & 1, ttsh::kWaitLimitNs)) atomicExch(a.err, 1);
      if (on) {
        const float2* g = gs + warp * n + k * piece;
        const float2* x = xs + (k % ring) * piece * CW + c;
        float2 u[2][8];
        float4 pq[2][4];
        auto fetch = [&](int s, int y) {
#pragma unroll
          for (int i = 0; i < 4; ++i) pq[s][i] = *reinterpret_cast<const float4*>(g + y + 2 * i);
#pragma unroll
          for (int i = 0; i < 8; ++i) u[s][i] = x[(y + i) * CW];
          asm volatile("" ::: "memory");   // loads stay ahead of the sums
        };
        auto sum = [&](int s, auto zero) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float2 v = u[s][i];
            const float p = i & 1 ? pq[s][i >> 1].z : pq[s][i >> 1].x, q = i & 1 ? pq[s][i >> 1].w : pq[s][i >> 1].y;
            const float p2 = decltype(zero)::value ? 1.f : p, q2 = decltype(zero)::value ? -0.f : -q;
            if constexpr (ADJ) {   // four sums, combined below
              ar[0] = fmaf(p, v.x, ar[0]);
              br[0] = fmaf(q, v.y, br[0]);
              ai[0] = fmaf(p, v.y, ai[0]);
              bi[0] = fmaf(q, v.x, bi[0]);
              ar[1] = fmaf(p2, v.x, ar[1]);
              br[1] = fmaf(q2, v.y, br[1]);
              ai[1] = fmaf(p2, v.y, ai[1]);
              bi[1] = fmaf(q2, v.x, bi[1]);
            } else {
              ar[0] = fmaf(p, v.x, fmaf(-q, v.y, ar[0]));
              ai[0] = fmaf(p, v.y, fmaf(q, v.x, ai[0]));
              ar[1] = fmaf(p2, v.x, fmaf(-q2, v.y, ar[1]));
              ai[1] = fmaf(p2, v.y, fmaf(q2, v.x, ai[1]));
            }
          }
        };
        auto sums = [&](auto zero) {
          fetch(0, 0);
#pragma unroll 1
          for (int y = 0; y < piece; y += 16) {   // a piece is a multiple of 16
            fetch(1, y + 8);
            sum(0, zero);
            fetch(0, y + 16 < piece ? y + 16 : 0);
            sum(1, zero);
          }
        };
        if (t0 + warp == 0) sums(std::true_type{});   // the pair (-m, 0)
        else sums(std::false_type{});
      }
      if (ring < pieces) {   // everybody is done with the piece
        __syncthreads();
        if (tid == 0 && k + ring < pieces) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // reads before the refill
          load_piece(k + ring);
        }
      }
    }
    if (on) {
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        if constexpr (ADJ) {
          ar[s] = ar[s] - br[s];
          ai[s] = ai[s] + bi[s];
        }
        hs[(2 * warp + s) * CW + c] = make_float2(ar[s], ai[s]);
        if (a.Hr) {
          const int j = s ? row_b(t0 + warp) : row_a(t0 + warp);
          const long long o = (((long long)b * J + j) * m + kx) * CW + c;
          a.Hr[o] = ar[s];
          a.Hi[o] = ai[s];
        }
      }
    }
  }
  __syncthreads();
  // ---- mixing of this block's modes: Y_o = sum_i W_io H_i with o = this lane, or in the adjoint
  // dH_i = sum_o conj(W_io) dY_o with i = this lane ----
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");   // the other blocks have started
  for (int jl = warp; jl < 2 * tn; jl += kColThreads / 32) {
    float sr = 0.f, si = 0.f;
    const __nv_bfloat16* w0 = wr + jl * WMAT;
    const __nv_bfloat16* w1 = wi + jl * WMAT;
#pragma unroll
    for (int i8 = 0; i8 < CW; i8 += 8) {
      __nv_bfloat16 pa[8], pb[8];
      if constexpr (ADJ) {
        *reinterpret_cast<uint4*>(pa) = *reinterpret_cast<const uint4*>(w0 + c * WROW + i8);
        *reinterpret_cast<uint4*>(pb) = *reinterpret_cast<const uint4*>(w1 + c * WROW + i8);
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          pa[i] = w0[(i8 + i) * CW + c];
          pb[i] = w1[(i8 + i) * CW + c];
        }
      }
      float4 h4[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) h4[i] = *reinterpret_cast<const float4*>(hs + jl * CW + i8 + 2 * i);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float p = __bfloat162float(pa[i]), q = __bfloat162float(pb[i]);
        const float u = i & 1 ? h4[i >> 1].z : h4[i >> 1].x, w = i & 1 ? h4[i >> 1].w : h4[i >> 1].y;
        if constexpr (ADJ) {
          sr = fmaf(p, u, fmaf(q, w, sr));
          si = fmaf(p, w, fmaf(-q, u, si));
        } else {
          sr = fmaf(p, u, fmaf(-q, w, sr));
          si = fmaf(p, w, fmaf(q, u, si));
        }
      }
    }
    // ---- into every block's copy of the mixed modes (distributed shared memory) ----
    const int t = t0 + (jl >> 1), j = jl & 1 ? row_b(t) : row_a(t);
    const uint32_t o0 = smem_u32(ys + j * CW + c);
#pragma unroll
    for (int r = 0; r < CS; ++r) {
      uint32_t d0;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d0) : "r"(o0), "r"(r));
      asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(d0), "f"(sr), "f"(si) : "memory");
    }
  }
  // every block's modes have arrived everywhere
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");

  // ---- Z_y = sum over j, in order: four y of two channels a thread ----
  const int c2 = 2 * (tid & 15);
  for (int yg = tid >> 4; yg < (y0 < n ? ny / 4 : 0); yg += kColThreads / 16) {
    float ar[2][4] = {}, ai[2][4] = {}, br[2][4] = {}, bi[2][4] = {};
#pragma unroll 4
    for (int j = 0; j < J; ++j) {
      const float4 p4 = *reinterpret_cast<const float4*>(vr + j * ny + 4 * yg);
      const float4 q4 = *reinterpret_cast<const float4*>(vi + j * ny + 4 * yg);
      const float4 yv = *reinterpret_cast<const float4*>(ys + j * CW + c2);
      const float pv[4] = {p4.x, p4.y, p4.z, p4.w}, qv[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const float u = s ? yv.z : yv.x, w = s ? yv.w : yv.y;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if constexpr (ADJ) {
            ar[s][i] = fmaf(pv[i], u, ar[s][i]);
            br[s][i] = fmaf(qv[i], w, br[s][i]);
            ai[s][i] = fmaf(pv[i], w, ai[s][i]);
            bi[s][i] = fmaf(qv[i], u, bi[s][i]);
          } else {   // conj(G) = Gr - i Gi
            ar[s][i] = fmaf(pv[i], u, fmaf(qv[i], w, ar[s][i]));
            ai[s][i] = fmaf(pv[i], w, fmaf(-qv[i], u, ai[s][i]));
          }
        }
      }
    }
    float* z0 = a.Z + (((long long)b * J + kx) * n + y0 + 4 * yg) * CW + c2;
    float* z1 = z0 + (long long)m * n * CW;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if constexpr (ADJ) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          ar[s][i] = ar[s][i] + br[s][i];
          ai[s][i] = ai[s][i] - bi[s][i];
        }
      }
      *reinterpret_cast<float2*>(z0 + i * CW) = make_float2(ar[0][i], ar[1][i]);
      *reinterpret_cast<float2*>(z1 + i * CW) = make_float2(ai[0][i], ai[1][i]);
    }
  }
}

// ---------------------------------------------------------------------------------------
// Gradients of the spectral weights: dW[i][o] = sum_b dY_o conj(H_i) per mode, b in order
// ---------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) mode_wgrad_kernel(const float* __restrict__ Hr, const float* __restrict__ Hi,
                                                         const float* __restrict__ dYr, const float* __restrict__ dYi,
                                                         int nmodes, int B, float* __restrict__ gWr, float* __restrict__ gWi) {
  const int mode = blockIdx.x, o4 = (threadIdx.x & 7) * 4, i = threadIdx.x >> 3;
  float ar[4] = {0, 0, 0, 0}, ai[4] = {0, 0, 0, 0};
  for (int b = 0; b < B; ++b) {
    const long long at = ((long long)b * nmodes + mode) * CW;
    const float hr = Hr[at + i], hi = Hi[at + i];
    const float4 p4 = *reinterpret_cast<const float4*>(dYr + at + o4), q4 = *reinterpret_cast<const float4*>(dYi + at + o4);
    const float p[4] = {p4.x, p4.y, p4.z, p4.w}, q[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      ar[k] = fmaf(p[k], hr, fmaf(q[k], hi, ar[k]));
      ai[k] = fmaf(q[k], hr, fmaf(-p[k], hi, ai[k]));
    }
  }
  const long long at = (long long)mode * CW * CW + i * CW + o4;
  *reinterpret_cast<float4*>(gWr + at) = make_float4(ar[0], ar[1], ar[2], ar[3]);
  *reinterpret_cast<float4*>(gWi + at) = make_float4(ai[0], ai[1], ai[2], ai[3]);
}

// ---------------------------------------------------------------------------------------
// Gradients of the channel-mixing weights: part[chunk][i * cd + o] = sum over the chunk's points
// of A[p][i] D[p][o], part[chunk][ca * cd + o] = sum of D[p][o].  A chunk is summed in groups of
// 64 points (in order inside a group, then the groups in order); a warp takes one group, whose
// 32 x 32 products it holds as 4 x 8 per lane, so that three 16-byte shared loads feed 32 FMAs;
// the next 32 points travel meanwhile.  At 524288 points: 39 us (134 MB, 20 us at the measured copy
// rate), where one output a thread with two shared loads for each FMA took 200 us.
// ---------------------------------------------------------------------------------------
enum WgA { WA_RAW = 0, WA_LIFT = 1, WA_X = 2 };       // rows of A: h as stored, x Wp + bp, x itself (4 wide)
enum WgD { WD_RAW = 0, WD_OUTER = 1, WD_ONE = 2 };              // rows of D: dz, dout Wq, dout itself (1 wide)

struct WgArgs {
  const float *A, *D;
  int a16;                // WA_LIFT, WA_X (the caller's x): 1 if it is 16-byte aligned
  const float *Wp, *bp;   // WA_LIFT
  const float* Wq;        // WD_OUTER
  long long P;
  int chunk;              // points per block
  float* part;            // [blocks][nout]
};

constexpr int kWgWarps = 4, kWgGroup = 64, kWgHalf = 32;
// per warp: two stages of 32 points of A and D (the group's sums take the second one's place at the
// end of a group, when nothing is on its way there); small inputs (x, dout) of the stages that
// are formed where they are read.  Three blocks fit an SM.
constexpr int kWgStage = kWgHalf * 2 * CW;
constexpr int kWgSmall = kWgHalf * 5;
constexpr int kWgSmem = kWgWarps * (2 * kWgStage + 2 * kWgSmall) * 4;

// 16 or 4 bytes global -> shared, zeros where `in` is false (src must be a valid address all the same)
__device__ __forceinline__ void cp_async16_or0(void* smem, const void* gmem, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(smem)), "l"(gmem), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async4_or0(void* smem, const void* gmem, bool in) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(smem)), "l"(gmem), "r"(in ? 4 : 0) : "memory");
}

template <int AM, int DM>
__global__ void __launch_bounds__(32 * kWgWarps) wgrad_kernel(WgArgs a) {
  constexpr int CA = AM == WA_X ? 4 : CW, CD = DM == WD_ONE ? 1 : CW;
  constexpr int NOUT = CA * CD + CD;
  constexpr int NACC = (NOUT + 32 * kWgWarps - 1) / (32 * kWgWarps);
  extern __shared__ __align__(16) float wg_sm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float* stage = wg_sm + warp * 2 * kWgStage;                              // [2][A 32 x 32 | D 32 x 32]
  float* small = wg_sm + kWgWarps * 2 * kWgStage + warp * 2 * kWgSmall;    // [2][x 32 x 4 | dout 32]
  float lw[5] = {0, 0, 0, 0, 0}, lq = 0.f;   // this lane's channel of the lift and of Wq
  if constexpr (AM == WA_LIFT) {
#pragma unroll
    for (int k = 0; k < 5; ++k) lw[k] = k < 4 ? a.Wp[k * CW + lane] : a.bp[lane];
  }
  if constexpr (DM == WD_OUTER) lq = a.Wq[lane];
  const long long c0 = (long long)blockIdx.x * a.chunk;
  const long long c1 = c0 + a.chunk < a.P ? c0 + a.chunk : a.P;
  // half h of the block's sequence: rounds of kWgWarps groups, two halves a group
  auto load = [&](int h) {
    const long long p0 = c0 + (long long)(h >> 1) * (kWgWarps * kWgGroup) + warp * kWgGroup + (h & 1) * kWgHalf;
    float* As = stage + (h & 1) * kWgStage;
    float* Ds = As + kWgHalf * CW;
    float* xs = small + (h & 1) * kWgSmall;
    if constexpr (AM == WA_RAW) {
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int e = lane + 32 * k;
        const bool in = p0 + (e >> 3) < c1;
        cp_async16_or0(As + e * 4, a.A + (in ? p0 * CW + e * 4 : 0), in);
      }
    } else {
      const bool in = p0 + lane < c1;
      const float* xp = a.A + (in ? (p0 + lane) * 4 : 0);
      if (a.a16) {
        cp_async16_or0(xs + lane * 4, xp, in);
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) cp_async4_or0(xs + lane * 4 + k, xp + k, in);
      }
    }
    if constexpr (DM == WD_RAW) {
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int e = lane + 32 * k;
        const bool in = p0 + (e >> 3) < c1;
        cp_async16_or0(Ds + e * 4, a.D + (in ? p0 * CW + e * 4 : 0), in);
      }
    } else {
      cp_async4_or0(xs + kWgHalf * 4 + lane, a.D + (p0 + lane < c1 ? p0 + lane : 0), p0 + lane < c1);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int rounds = (int)((c1 - c0 + kWgWarps * kWgGroup - 1) / (kWgWarps * kWgGroup));
  float acc[NACC];
#pragma unroll
  for (int k = 0; k < NACC; ++k) acc[k] = 0.f;
  load(0);
  for (int rd = 0; rd < rounds; ++rd) {
    // ---- this warp's group of 64 points, in order ----
    const int ig = (lane >> 2) * 4, og = (lane & 3) * 8;
    constexpr int NI = CD == 1 ? 1 : 4, NO = CD == 1 || CA == 4 ? 1 : 8;
    float s[NI][NO], bsum = 0.f;
#pragma unroll
    for (int i = 0; i < NI; ++i)
#pragma unroll
      for (int o = 0; o < NO; ++o) s[i][o] = 0.f;
#pragma unroll 1
    for (int hf = 0; hf < 2; ++hf) {
      const int h = 2 * rd + hf;
      if (h + 1 < 2 * rounds) load(h + 1);
      else asm volatile("cp.async.commit_group;" ::: "memory");
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      __syncwarp();
      float* As = stage + hf * kWgStage;
      float* Ds = As + kWgHalf * CW;
      const float* xs = small + hf * kWgSmall;
      const long long p0 = c0 + (long long)rd * (kWgWarps * kWgGroup) + warp * kWgGroup + hf * kWgHalf;
      if constexpr (AM == WA_LIFT) {   // lane = channel
        const int live = c1 - p0 < kWgHalf ? (int)(c1 - p0) : kWgHalf;
#pragma unroll 8
        for (int r = 0; r < kWgHalf; ++r) {
          const float4 xv = *reinterpret_cast<const float4*>(xs + 4 * r);
          const float h = fmaf(xv.w, lw[3], fmaf(xv.z, lw[2], fmaf(xv.y, lw[1], fmaf(xv.x, lw[0], lw[4]))));
          As[r * CW + lane] = r < live ? h : 0.f;
        }
      }
      if constexpr (DM == WD_OUTER) {
#pragma unroll
        for (int r = 0; r < kWgHalf; r += 4) {
          const float4 d4 = *reinterpret_cast<const float4*>(xs + kWgHalf * 4 + r);
          Ds[r * CW + lane] = d4.x * lq;
          Ds[(r + 1) * CW + lane] = d4.y * lq;
          Ds[(r + 2) * CW + lane] = d4.z * lq;
          Ds[(r + 3) * CW + lane] = d4.w * lq;
        }
      }
      if constexpr (AM == WA_LIFT || DM == WD_OUTER) __syncwarp();
      if constexpr (CD == 1) {          // lane = i
#pragma unroll 8
        for (int r = 0; r < kWgHalf; ++r) {
          const float d = xs[kWgHalf * 4 + r];
          s[0][0] = fmaf(As[r * CW + lane], d, s[0][0]);
          bsum += d;
        }
      } else if constexpr (CA == 4) {   // lane = o
#pragma unroll 8
        for (int r = 0; r < kWgHalf; ++r) {
          const float4 x4 = *reinterpret_cast<const float4*>(xs + 4 * r);
          const float d = Ds[r * CW + lane];
          s[0][0] = fmaf(x4.x, d, s[0][0]);
          s[1][0] = fmaf(x4.y, d, s[1][0]);
          s[2][0] = fmaf(x4.z, d, s[2][0]);
          s[3][0] = fmaf(x4.w, d, s[3][0]);
          bsum += d;
        }
      } else {
#pragma unroll 4
        for (int r = 0; r < kWgHalf; ++r) {
          const float4 a4 = *reinterpret_cast<const float4*>(As + r * CW + ig);
          const float4 d4 = *reinterpret_cast<const float4*>(Ds + r * CW + og);
          const float4 e4 = *reinterpret_cast<const float4*>(Ds + r * CW + og + 4);
          bsum += Ds[r * CW + lane];
          const float av[4] = {a4.x, a4.y, a4.z, a4.w};
          const float dv[8] = {d4.x, d4.y, d4.z, d4.w, e4.x, e4.y, e4.z, e4.w};
#pragma unroll
          for (int i = 0; i < NI; ++i)
#pragma unroll
            for (int o = 0; o < NO; ++o) s[i][o] = fmaf(av[i], dv[o], s[i][o]);
        }
      }
      __syncwarp();   // read before the next load into this stage
    }
    float* S = stage + kWgStage;
    if constexpr (CD == 1) {
      S[lane] = s[0][0];
      if (lane == 0) S[CW] = bsum;
    } else if constexpr (CA == 4) {
#pragma unroll
      for (int i = 0; i < 4; ++i) S[i * CW + lane] = s[i][0];
      S[4 * CW + lane] = bsum;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int o = 0; o < NO; o += 4)
          *reinterpret_cast<float4*>(S + (ig + i) * CW + og + o) = make_float4(s[i][o], s[i][o + 1], s[i][o + 2], s[i][o + 3]);
      S[CW * CW + lane] = bsum;
    }
    __syncthreads();
    // ---- groups in order ----
    for (int w = 0; w < kWgWarps && c0 + ((long long)rd * kWgWarps + w) * kWgGroup < c1; ++w) {
#pragma unroll
      for (int k = 0; k < NACC; ++k) {
        const int o = tid + k * 32 * kWgWarps;
        if (o < NOUT) acc[k] += wg_sm[(2 * w + 1) * kWgStage + o];
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int k = 0; k < NACC; ++k) {
    const int o = tid + k * 32 * kWgWarps;
    if (o < NOUT) a.part[(long long)blockIdx.x * NOUT + o] = acc[k];
  }
}

// Sums of the blocks' partials in double: 8 outputs x 32 slices of the blocks per block; blockIdx.y
// selects the gradient.
struct WgReduce {
  const float* part;
  float *gw, *gb;
  int nout, nw;   // outputs, of which the first nw go to gw and the others to gb
};
constexpr int kMaxWg = 18;   // layers + 2
struct WgReduceAll {
  WgReduce g[kMaxWg];
  int nblk;
};

__global__ void __launch_bounds__(256) wgrad_reduce_all_kernel(const __grid_constant__ WgReduceAll a) {
  __shared__ double red[32][9];
  const WgReduce& g = a.g[blockIdx.y];
  const int ol = threadIdx.x & 7, sl = threadIdx.x >> 3, o = blockIdx.x * 8 + ol;
  if (blockIdx.x * 8 >= g.nout) return;
  const int per = (a.nblk + 31) / 32, b0 = sl * per, b1 = b0 + per < a.nblk ? b0 + per : a.nblk;
  double s = 0.0;
  if (o < g.nout)
    for (int b = b0; b < b1; ++b) s += g.part[(long long)b * g.nout + o];
  red[sl][ol] = s;
  __syncthreads();
  if (threadIdx.x < 8 && o < g.nout) {
    double t = 0.0;
    for (int i = 0; i < 32; ++i) t += red[i][ol];
    if (o < g.nw) g.gw[o] = (float)t;
    else g.gb[o - g.nw] = (float)t;
  }
}

// Loss from the grid rows' sums of squares (fixed order).
__global__ void __launch_bounds__(256) loss_kernel(const double* __restrict__ part, long long Q, double inv, double* __restrict__ loss) {
  __shared__ double red[256];
  double s = 0.0;
  for (long long q = threadIdx.x; q < Q; q += 256) s += part[q];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int k = 128; k >= 1; k >>= 1) {
    if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
    __syncthreads();
  }
  if (threadIdx.x == 0) *loss = red[0] * inv;
}

}  // namespace fno_dev

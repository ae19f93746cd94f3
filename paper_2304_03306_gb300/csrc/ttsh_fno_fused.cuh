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
// Spectral columns lie as [b][k][y][channel] (k = Re kx 0..m-1, then Im), so that a block's two
// columns are contiguous.  Every FP32 sum runs in the order of the separate kernels these
// replace, so that results, including every rounding to BF16, are the same bits.
#pragma once

namespace fno_dev {

__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_all;\n" ::: "memory");
}

// ---------------------------------------------------------------------------------------
// Row kernel
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
  const __nv_bfloat16* C;    // [32][n]: matrix that contracts the row to the kept kx
  float* X;                  // [B][J][n][32]: contracted columns
  const float* bias;         // 32
  const float* x;            // R_LIFT: [P][4]
  const float *Wp, *bp;      // R_LIFT
  const float* zin;          // R_BWD: z of the layer below
  float* zout;               // forward in training: z (null otherwise)
  __nv_bfloat16* hb;         // result in BF16: h_{l+1}, or dz
  float* dz;                 // R_BWD: dz', R_BWD_FIRST: dh
  const float *Wq, *bq;      // R_LAST*
  float* out;                // R_LAST*: [P]
  const float* target;       // R_LAST_TRAIN: [P]
  float* dout;               // R_LAST_TRAIN: [P]
  double* lpart;             // R_LAST_TRAIN: sum of squared errors of each grid row
  int n, J;
  long long Q, P;            // grid rows, points
  int* err;
};

__host__ __device__ constexpr bool row_has_mma(int mode) { return mode != R_LIFT; }
__host__ __device__ constexpr bool row_contracts(int mode) { return mode != R_LAST && mode != R_BWD_FIRST; }
__host__ __device__ constexpr bool row_stages(int mode, bool train) {   // FP32 rows through shared memory
  return mode == R_BWD || mode == R_BWD_FIRST || mode == R_LAST_TRAIN || (mode == R_FWD && train);
}

// Dynamic shared memory: A tile | C | E | W | Z operand | FP32 rows of every warp, and 128 bytes
// to align the base.
inline int row_smem(int mode, bool train, int n) {
  const int nr = n < 128 ? 128 : n;
  return 128 + nr * 64 + 64 * n + 2048 + (row_has_mma(mode) ? nr * 64 + 2048 : 0) +
         (row_stages(mode, train) ? nr * 128 : 0);
}

// 16-byte piece i of row r in a warp's 32 x 128-byte block, rotated so that both a thread's own
// row and a warp's consecutive pieces meet every bank once.
__device__ __forceinline__ float4* row_piece(unsigned char* blk, int r, int i) {
  return reinterpret_cast<float4*>(blk + r * 128 + ((i ^ (r & 7)) << 4));
}

template <int MODE, int T, bool TRAIN>
__global__ void __launch_bounds__(128 * T) row_layer_kernel(RowArgs a) {
  constexpr int NT = 128 * T;
  constexpr int TCOLS = 64 * T;   // per x tile: 32 columns for the channel mixing, 32 for the expansion
  extern __shared__ __align__(16) unsigned char row_dyn[];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_base;
  __shared__ float sc[CW * 6];    // bias / Wp, bp / Wq
  __shared__ double lred[4 * T];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = a.n, J = a.J, nr = n < 128 ? 128 : n;
  unsigned char* base = row_dyn + ((128u - (smem_u32(row_dyn) & 127u)) & 127u);
  unsigned char* sA = base;
  unsigned char* sC = sA + nr * 64;
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
  cp_async_wait();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
  const int tile = warp >> 2;
  const int x = tid;               // this thread's point of the grid row
  const bool live = x < n;
  const int wrows = n - warp * 32 >= 32 ? 32 : (n - warp * 32 > 0 ? n - warp * 32 : 0);
  uint32_t phase = 0;
  pdl_wait();
  pdl_launch();

  for (long long q = blockIdx.x; q < a.Q; q += gridDim.x) {
    const long long p0 = q * n;
    const int b = (int)(q / n), y = (int)(q - (long long)b * n);
    uint32_t acc[CW];
    float v[CW];
    if constexpr (row_has_mma(MODE)) {
      for (int c = tid; c < n * 4; c += NT) cp_async16(sA + core_off(c >> 2, c & 3), a.A + p0 * CW + c * 8);
      if constexpr (MODE == R_BWD) {   // z of the layer below, for GELU'
        for (int i = lane; i < wrows * 8; i += 32)
          cp_async16(row_piece(blk, i >> 3, i & 7), a.zin + (p0 + warp * 32) * CW + i * 4);
      }
      // columns to expand as the K-major operand [channel][k]: eight k of one channel a thread
      if (warp < 4) {
        __nv_bfloat16 e[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int j = warp * 8 + i;
          const float f = j < J ? a.Z[(((long long)b * J + j) * n + y) * CW + lane] : 0.f;
          e[i] = __float2bfloat16_rn(f);
        }
        *reinterpret_cast<uint4*>(sZ + core_off(lane, warp)) = *reinterpret_cast<const uint4*>(e);
      }
      cp_async_wait();
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
      const bool done = ttsh::mbar_wait_bounded(smem_u32(&mbar), phase, ttsh::kWaitLimitNs);
      if (__syncthreads_or(!done)) {
        if (tid == 0) atomicExch(a.err, 1);
        break;
      }
      phase ^= 1u;
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
      const float4 xv = live ? *reinterpret_cast<const float4*>(a.x + (p0 + x) * 4) : make_float4(0, 0, 0, 0);
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
    if constexpr ((MODE == R_FWD && TRAIN) || MODE == R_LAST_TRAIN) {
      put_rows();
      store_rows(a.zout);
    }
    if constexpr (MODE == R_FWD) {
#pragma unroll
      for (int c = 0; c < CW; ++c) v[c] = gelu(v[c]);
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
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 z = *row_piece(blk, lane, i);
        v[4 * i] *= gelu_grad(z.x);
        v[4 * i + 1] *= gelu_grad(z.y);
        v[4 * i + 2] *= gelu_grad(z.z);
        v[4 * i + 3] *= gelu_grad(z.w);
      }
    }
    if constexpr (MODE == R_BWD || MODE == R_BWD_FIRST) {
      if constexpr (MODE == R_BWD) __syncwarp();
      put_rows();
      store_rows(a.dz);
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
        float* xo = a.X + ((long long)b * J * n + y) * CW + lane;
#pragma unroll
        for (int j = 0; j < CW; ++j)
          if (j < J) xo[(long long)j * n * CW] = __uint_as_float(acc[j]);
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");   // accumulators read before reuse
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) tc_dealloc(tmem, TCOLS);
}

// ---------------------------------------------------------------------------------------
// Column kernel
// ---------------------------------------------------------------------------------------
struct ColArgs {
  const float* X;                      // [B][J][n][32]
  const float *Gr, *Gi;                // [J][n]: exp(-2 pi i ky y / n)
  const __nv_bfloat16 *Wr, *Wi;        // [J][m][32][32]
  float *Hr, *Hi;                      // [B][J][m][32]: modes before the mixing (null: not kept)
  float* Z;                            // [B][J][n][32]
  int n, m;
  int* err;
};

// Forward (ADJ = false): H_j = sum_y G_jy X_y, Y = W H per mode, Z_y = sum_j conj(G_jy) Y_j.
// Adjoint: the same transforms around dH = W^H dY.  Block `rank` of the cluster transforms JB of
// the kept ky and JB's share of the mixing, and afterwards n / CS values of y.
constexpr int kColThreads = 256;
// BF16 values between the rows of a staged 32 x 32 weight: the adjoint reads a row per lane in
// 16-byte pieces, and 80 bytes apart eight of them meet every bank once.
__host__ __device__ constexpr int col_wrow(bool adj) { return adj ? 40 : CW; }

inline int col_smem(int n, int J, int CS) {
  const int JB = (J + CS - 1) / CS, ny = n / CS;
  return 128 + 2 * n * CW * 4 + 2 * JB * n * 4 + 2 * J * ny * 4 + 2 * JB * CW * col_wrow(true) * 2 + 4 * JB * CW * 4 + 2 * J * CW * 4;
}

template <int CS, bool ADJ>
__global__ void __launch_bounds__(kColThreads) column_layer_kernel(ColArgs a) {
  extern __shared__ __align__(16) unsigned char col_dyn[];
  __shared__ __align__(8) uint64_t mbar;
  const int tid = threadIdx.x, warp = tid >> 5, c = tid & 31;
  const int n = a.n, m = a.m, J = 2 * m;
  const int kx = blockIdx.x / CS, rank = blockIdx.x % CS, b = blockIdx.y;
  const int JB = (J + CS - 1) / CS, ny = n / CS;
  const int j0 = rank * JB, jn = J - j0 < JB ? (J - j0 > 0 ? J - j0 : 0) : JB;   // this block's ky rows
  const int y0 = rank * ny;
  constexpr int WROW = col_wrow(ADJ), WMAT = CW * WROW;
  unsigned char* base = col_dyn + ((128u - (smem_u32(col_dyn) & 127u)) & 127u);
  float* xr = reinterpret_cast<float*>(base);                 // [n][32]
  float* xi = xr + n * CW;
  float* gr = xi + n * CW;                                    // [JB][n]
  float* gi = gr + JB * n;
  float* vr = gi + JB * n;                                    // [J][ny]: this block's y of every ky row
  float* vi = vr + J * ny;
  float* yr = vi + J * ny;                                    // [J][32]: every mixed mode
  float* yi = yr + J * CW;
  float* hr = yi + J * CW;                                    // [JB][32]: this block's modes
  float* hi = hr + JB * CW;
  float* mr = hi + JB * CW;                                   // [JB][32]: the same, mixed
  float* mi = mr + JB * CW;
  __nv_bfloat16* wr = reinterpret_cast<__nv_bfloat16*>(mi + JB * CW);   // [JB][32][WROW]
  __nv_bfloat16* wi = wr + JB * WMAT;

  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int e = tid; e < jn * n / 4; e += kColThreads) {
    cp_async16(gr + 4 * e, a.Gr + (long long)j0 * n + 4 * e);
    cp_async16(gi + 4 * e, a.Gi + (long long)j0 * n + 4 * e);
  }
  for (int e = tid; e < J * ny / 4; e += kColThreads) {
    const int j = e / (ny / 4), r = e % (ny / 4);
    cp_async16(vr + 4 * e, a.Gr + (long long)j * n + y0 + 4 * r);
    cp_async16(vi + 4 * e, a.Gi + (long long)j * n + y0 + 4 * r);
  }
  for (int e = tid; e < jn * (CW * CW / 8); e += kColThreads) {
    const int jl = e / (CW * CW / 8), r = e % (CW * CW / 8);
    const long long src = ((long long)(j0 + jl) * m + kx) * CW * CW + 8 * r;
    const int dst = jl * WMAT + (r >> 2) * WROW + 8 * (r & 3);
    cp_async16(wr + dst, a.Wr + src);
    cp_async16(wi + dst, a.Wi + src);
  }
  __syncthreads();   // the barrier is initialised
  pdl_wait();
  pdl_launch();
  if (tid == 0) {
    const uint32_t bytes = (uint32_t)(n * CW * 4);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&mbar)), "r"(2 * bytes) : "memory");
    const float* s0 = a.X + ((long long)b * J + kx) * n * CW;
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(xr)), "l"(s0), "r"(bytes), "r"(smem_u32(&mbar)) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(xi)), "l"(s0 + (long long)m * n * CW), "r"(bytes), "r"(smem_u32(&mbar)) : "memory");
  }
  cp_async_wait();
  if (!ttsh::mbar_wait_bounded(smem_u32(&mbar), 0, ttsh::kWaitLimitNs)) atomicExch(a.err, 1);
  __syncthreads();

  for (int jl = warp; jl < jn; jl += kColThreads / 32) {
    // ---- H_j = sum over y, in order ----
    float ar = 0.f, ai = 0.f, br = 0.f, bi = 0.f;
    const float* g0 = gr + jl * n;
    const float* g1 = gi + jl * n;
#pragma unroll 2
    for (int y = 0; y < n; y += 4) {
      const float4 p4 = *reinterpret_cast<const float4*>(g0 + y), q4 = *reinterpret_cast<const float4*>(g1 + y);
      const float pv[4] = {p4.x, p4.y, p4.z, p4.w}, qv[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float u = xr[(y + i) * CW + c], w = xi[(y + i) * CW + c];
        if constexpr (ADJ) {   // four sums, combined below
          ar = fmaf(pv[i], u, ar);
          br = fmaf(qv[i], w, br);
          ai = fmaf(pv[i], w, ai);
          bi = fmaf(qv[i], u, bi);
        } else {
          ar = fmaf(pv[i], u, fmaf(-qv[i], w, ar));
          ai = fmaf(pv[i], w, fmaf(qv[i], u, ai));
        }
      }
    }
    if constexpr (ADJ) {
      ar = ar - br;
      ai = ai + bi;
    }
    hr[jl * CW + c] = ar;
    hi[jl * CW + c] = ai;
    if (a.Hr) {
      const long long o = (((long long)b * J + j0 + jl) * m + kx) * CW + c;
      a.Hr[o] = ar;
      a.Hi[o] = ai;
    }
    __syncwarp();
    // ---- mixing of this mode ----
    float sr = 0.f, si = 0.f;
    const __nv_bfloat16* w0 = wr + jl * WMAT;
    const __nv_bfloat16* w1 = wi + jl * WMAT;
    if constexpr (ADJ) {   // dH_i = sum_o conj(W_io) dY_o, i = this lane
#pragma unroll
      for (int o8 = 0; o8 < CW; o8 += 8) {
        const uint4 a4 = *reinterpret_cast<const uint4*>(w0 + c * WROW + o8);
        const uint4 b4 = *reinterpret_cast<const uint4*>(w1 + c * WROW + o8);
        const __nv_bfloat16* pa = reinterpret_cast<const __nv_bfloat16*>(&a4);
        const __nv_bfloat16* pb = reinterpret_cast<const __nv_bfloat16*>(&b4);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float p = __bfloat162float(pa[i]), q = __bfloat162float(pb[i]);
          const float u = hr[jl * CW + o8 + i], w = hi[jl * CW + o8 + i];
          sr = fmaf(p, u, fmaf(q, w, sr));
          si = fmaf(p, w, fmaf(-q, u, si));
        }
      }
    } else {               // Y_o = sum_i W_io H_i, o = this lane
#pragma unroll 8
      for (int i = 0; i < CW; ++i) {
        const float p = __bfloat162float(w0[i * CW + c]), q = __bfloat162float(w1[i * CW + c]);
        const float u = hr[jl * CW + i], w = hi[jl * CW + i];
        sr = fmaf(p, u, fmaf(-q, w, sr));
        si = fmaf(p, w, fmaf(q, u, si));
      }
    }
    mr[jl * CW + c] = sr;
    mi[jl * CW + c] = si;
  }

  // ---- every block's mixed modes, through distributed shared memory ----
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
  for (int e = tid; e < J * CW / 4; e += kColThreads) {
    const int j = e / (CW / 4), r = j / JB;
    const int off = ((j - r * JB) * CW + 4 * (e % (CW / 4))) * 4;
    uint32_t s0, s1;
    float4 p, q;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(s0) : "r"(smem_u32(mr) + off), "r"(r));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(s1) : "r"(smem_u32(mi) + off), "r"(r));
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(p.x), "=f"(p.y), "=f"(p.z), "=f"(p.w) : "r"(s0) : "memory");
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(q.x), "=f"(q.y), "=f"(q.z), "=f"(q.w) : "r"(s1) : "memory");
    *reinterpret_cast<float4*>(yr + 4 * e) = p;
    *reinterpret_cast<float4*>(yi + 4 * e) = q;
  }
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");   // done with the other blocks' memory
  __syncthreads();

  // ---- Z_y = sum over j, in order, four y a thread ----
  float* z0 = a.Z + (((long long)b * J + kx) * n + y0) * CW + c;
  float* z1 = z0 + (long long)m * n * CW;
  for (int yg = warp; yg < ny / 4; yg += kColThreads / 32) {
    float ar[4] = {0, 0, 0, 0}, ai[4] = {0, 0, 0, 0}, br[4] = {0, 0, 0, 0}, bi[4] = {0, 0, 0, 0};
#pragma unroll 4
    for (int j = 0; j < J; ++j) {
      const float4 p4 = *reinterpret_cast<const float4*>(vr + j * ny + 4 * yg);
      const float4 q4 = *reinterpret_cast<const float4*>(vi + j * ny + 4 * yg);
      const float pv[4] = {p4.x, p4.y, p4.z, p4.w}, qv[4] = {q4.x, q4.y, q4.z, q4.w};
      const float u = yr[j * CW + c], w = yi[j * CW + c];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if constexpr (ADJ) {
          ar[i] = fmaf(pv[i], u, ar[i]);
          br[i] = fmaf(qv[i], w, br[i]);
          ai[i] = fmaf(pv[i], w, ai[i]);
          bi[i] = fmaf(qv[i], u, bi[i]);
        } else {   // conj(G) = Gr - i Gi
          ar[i] = fmaf(pv[i], u, fmaf(qv[i], w, ar[i]));
          ai[i] = fmaf(pv[i], w, fmaf(-qv[i], u, ai[i]));
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if constexpr (ADJ) {
        ar[i] = ar[i] + br[i];
        ai[i] = ai[i] - bi[i];
      }
      z0[(4 * yg + i) * CW] = ar[i];
      z1[(4 * yg + i) * CW] = ai[i];
    }
  }
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
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
// 32 x 32 products it holds as 4 x 8 per lane, so that three 16-byte shared loads feed 32 FMAs.
// ---------------------------------------------------------------------------------------
enum WgA { WA_RAW = 0, WA_GELU = 1, WA_LIFT = 2, WA_X = 3 };    // rows of A: z, GELU(z), x Wp + bp, x itself (4 wide)
enum WgD { WD_RAW = 0, WD_OUTER = 1, WD_ONE = 2 };              // rows of D: dz, dout Wq, dout itself (1 wide)

struct WgArgs {
  const float *A, *D;
  const float *Wp, *bp;   // WA_LIFT
  const float* Wq;        // WD_OUTER
  long long P;
  int chunk;              // points per block
  float* part;            // [blocks][nout]
};

constexpr int kWgWarps = 4, kWgGroup = 64;
constexpr int kWgSmem = kWgWarps * kWgGroup * 2 * CW * 4;

template <int AM, int DM>
__global__ void __launch_bounds__(32 * kWgWarps) wgrad_kernel(WgArgs a) {
  constexpr int CA = AM == WA_X ? 4 : CW, CD = DM == WD_ONE ? 1 : CW;
  constexpr int NOUT = CA * CD + CD;
  constexpr int NACC = (NOUT + 32 * kWgWarps - 1) / (32 * kWgWarps);
  extern __shared__ __align__(16) float wg_sm[];
  __shared__ float sp[5 * CW];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float* As = wg_sm + warp * kWgGroup * 2 * CW;   // [64][32]
  float* Ds = As + kWgGroup * CW;                 // [64][32]
  if constexpr (AM == WA_LIFT) {
    for (int i = tid; i < 5 * CW; i += 32 * kWgWarps) sp[i] = i < 4 * CW ? a.Wp[i] : a.bp[i - 4 * CW];
    __syncthreads();
  }
  const long long c0 = (long long)blockIdx.x * a.chunk;
  const long long c1 = c0 + a.chunk < a.P ? c0 + a.chunk : a.P;
  float acc[NACC];
#pragma unroll
  for (int k = 0; k < NACC; ++k) acc[k] = 0.f;
  for (long long g0 = c0; g0 < c1; g0 += (long long)kWgWarps * kWgGroup) {
    const long long p0 = g0 + warp * kWgGroup;
    // ---- this warp's group: rows of A and D (zero past the chunk) ----
    if constexpr (AM == WA_RAW || AM == WA_GELU) {
#pragma unroll 8
      for (int e = lane; e < kWgGroup * CW / 4; e += 32) {
        float4 z = make_float4(0, 0, 0, 0);
        if (p0 + (e >> 3) < c1) {
          z = *reinterpret_cast<const float4*>(a.A + p0 * CW + e * 4);
          if constexpr (AM == WA_GELU) z = make_float4(gelu(z.x), gelu(z.y), gelu(z.z), gelu(z.w));
        }
        *reinterpret_cast<float4*>(As + e * 4) = z;
      }
    } else {
#pragma unroll
      for (int h = 0; h < kWgGroup / 32; ++h) {
        const int r = h * 32 + lane;
        const bool in = p0 + r < c1;
        const float4 xv = in ? *reinterpret_cast<const float4*>(a.A + (p0 + r) * 4) : make_float4(0, 0, 0, 0);
        if constexpr (AM == WA_X) {
          *reinterpret_cast<float4*>(As + r * CW) = xv;
        } else {
#pragma unroll
          for (int c = 0; c < CW; ++c) {   // column rotated by the row: no two lanes on one bank
            const int cc = (c + lane) & 31;
            As[r * CW + cc] = in ? fmaf(xv.w, sp[3 * CW + cc], fmaf(xv.z, sp[2 * CW + cc],
                                   fmaf(xv.y, sp[CW + cc], fmaf(xv.x, sp[cc], sp[4 * CW + cc])))) : 0.f;
          }
        }
      }
    }
    if constexpr (DM == WD_RAW) {
#pragma unroll 8
      for (int e = lane; e < kWgGroup * CW / 4; e += 32) {
        float4 z = make_float4(0, 0, 0, 0);
        if (p0 + (e >> 3) < c1) z = *reinterpret_cast<const float4*>(a.D + p0 * CW + e * 4);
        *reinterpret_cast<float4*>(Ds + e * 4) = z;
      }
    } else {
#pragma unroll
      for (int h = 0; h < kWgGroup / 32; ++h) {
        const int r = h * 32 + lane;
        Ds[r * (DM == WD_ONE ? 1 : CW)] = p0 + r < c1 ? a.D[p0 + r] : 0.f;
      }
      if constexpr (DM == WD_OUTER) {
        __syncwarp();
        const float w = a.Wq[lane];
        for (int r = 0; r < kWgGroup; ++r) {
          const float g = Ds[r * CW];
          __syncwarp();
          Ds[r * CW + lane] = g * w;
        }
      }
    }
    __syncwarp();
    // ---- the group's sums, r in order ----
    float bsum = 0.f;
    if constexpr (CD == 1) {
      float s = 0.f;
#pragma unroll 8
      for (int r = 0; r < kWgGroup; ++r) {
        const float d = Ds[r];
        s = fmaf(As[r * CW + lane], d, s);
        bsum += d;
      }
      __syncwarp();
      As[lane] = s;
      if (lane == 0) As[CW] = bsum;
    } else if constexpr (CA == 4) {
      float s[4] = {0, 0, 0, 0};   // lane = o
#pragma unroll 8
      for (int r = 0; r < kWgGroup; ++r) {
        const float4 x4 = *reinterpret_cast<const float4*>(As + r * CW);
        const float d = Ds[r * CW + lane];
        s[0] = fmaf(x4.x, d, s[0]);
        s[1] = fmaf(x4.y, d, s[1]);
        s[2] = fmaf(x4.z, d, s[2]);
        s[3] = fmaf(x4.w, d, s[3]);
        bsum += d;
      }
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 4; ++i) As[i * CW + lane] = s[i];
      As[4 * CW + lane] = bsum;
    } else {
      const int ig = (lane >> 2) * 4, og = (lane & 3) * 8;
      float s[4][8];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int o = 0; o < 8; ++o) s[i][o] = 0.f;
#pragma unroll 4
      for (int r = 0; r < kWgGroup; ++r) {
        const float4 a4 = *reinterpret_cast<const float4*>(As + r * CW + ig);
        const float4 d4 = *reinterpret_cast<const float4*>(Ds + r * CW + og);
        const float4 e4 = *reinterpret_cast<const float4*>(Ds + r * CW + og + 4);
        bsum += Ds[r * CW + lane];
        const float av[4] = {a4.x, a4.y, a4.z, a4.w};
        const float dv[8] = {d4.x, d4.y, d4.z, d4.w, e4.x, e4.y, e4.z, e4.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int o = 0; o < 8; ++o) s[i][o] = fmaf(av[i], dv[o], s[i][o]);
      }
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int o = 0; o < 8; ++o) As[(ig + i) * CW + og + o] = s[i][o];
      As[CW * CW + lane] = bsum;
    }
    __syncthreads();
    // ---- groups in order ----
    for (int w = 0; w < kWgWarps && g0 + w * kWgGroup < c1; ++w) {
      const float* S = wg_sm + w * kWgGroup * 2 * CW;
#pragma unroll
      for (int k = 0; k < NACC; ++k) {
        const int o = tid + k * 32 * kWgWarps;
        if (o < NOUT) acc[k] += S[o];
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

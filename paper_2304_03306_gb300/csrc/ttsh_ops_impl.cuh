// ttsh_ops_impl.cuh - template launchers; included by the per-precision translation units,
// each of which defines TTSH_T (float or double), TTSH_REGISTRY (function name) and
// TTSH_SIZES (an X-macro list of the grid sizes it instantiates).
#pragma once

#include <atomic>
#include <cstring>

#include "ttsh_args.cuh"

namespace ttsh {

template <typename K>
static cudaError_t set_smem(K kernel, int bytes, std::atomic<int>& done) {
  if (done.load(std::memory_order_acquire)) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) done.store(1, std::memory_order_release);
  return e;
}

// Shared memory that the widest reservation of spread_smem takes; every step kernel allows it.
constexpr int kSpreadSmem = 116 * 1024;

static int sm_count() {
  static std::atomic<int> sms{0};
  int v = sms.load(std::memory_order_acquire);
  if (v == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      v = 1 << 30;
    sms.store(v, std::memory_order_release);
  }
  return v;
}

// Shared memory that a programmatic dependent launch of at most one block per SM reserves per block,
// so that blocks admitted early (while the previous pass still runs) cannot pile up on the SMs
// that are free first and leave others idle when they start.  More than half an SM's keeps
// every other block off it, those of domains stepped on streams of their own among them, so it
// is left to a float 512^2 domain that was asked or tuned to overlap (us a step: one domain 9.5
// reserved, 10.2 without; eight domains 44.4 and 25.8 a step of all, ordinary launches 29.2).
// Double takes what leaves room for a second block from 256^2 (256^2: one domain 35.1 and 46.4
// without, eight 137.5 and 136.9; with half an SM's 35.1 and 143.8) and for two more below
// (128^2: one domain 20.3 and 24.4, eight 37.5 and 42.3; half an SM's 20.6 and 73.2).  Float up to
// 128^2 takes a quarter of an SM's (64^2: one domain 6.06 and 6.09, thirty-two 14.8 and 15.2; half
// an SM's 6.06 and 19.3); at 256^2 it gains nothing (one domain 7.2 either way, sixteen 14.8
// without and 42.9 with half an SM's, where ordinary launches take 17.4).
template <typename T, int N>
static int spread_smem(const DomainDev& d) {
  if (sizeof(T) == 8) return (N >= 256 ? 92 : 73) * 1024;
  return N <= 128 ? 54 * 1024 : N == 512 && d.pdl == 1 ? kSpreadSmem : 0;
}

// Dynamic shared memory of a step-pass launch: the pass's own, or `spread` for a launch of at most
// one block per SM.
static int launch_smem(int smem, int grid, int spread) {
  return smem < spread && grid <= sm_count() ? spread : smem;
}

// Whether launches on this stream go into a graph - the library's own, a corrected rollout's or the
// caller's: the stream is asked, so that no capture has to say so.
static bool capturing(cudaStream_t s) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &st) == cudaSuccess) return st != cudaStreamCaptureStatusNone;
  cudaGetLastError();   // (the legacy stream beside another's capture: the launch itself reports it)
  return false;
}

// Step kernels use programmatic dependent launch as the launch mode says; while none is set, where it
// pays (results are the same bits): when they are launched one by one, and in graphs on grids up
// to 512^2.  One by one the overlap hides the gap between launches (us a step: 256^2 float 12.0 ->
// 7.8, 1024^2 26.8 -> 23.4, 2048^2 87.2 -> 81.9); in a graph it saves 0.5 us of a small grid's pass
// (256^2 8.47 -> 7.34 us a step, 512^2 10.99 -> 9.81, 512^2 double 95.7 -> 94.1) but costs at
// 1024^2 (22.7 -> 23.8) and does nothing beyond.
template <int N>
static bool step_pdl(const DomainDev& d, cudaStream_t s) {
  if (d.whole) return false;
  return d.pdl == kPdlAuto ? N <= kPdlMaxN || !capturing(s) : d.pdl != 0;
}

// Launch, optionally as a programmatic dependent launch (the kernel may start while the
// previous kernel in the stream is still running; it waits (griddepcontrol.wait) before it
// touches anything that kernel writes) and optionally in clusters of `cl` blocks along x.
template <typename... P, typename... V>
static cudaError_t launch_k(void (*kernel)(P...), int grid, int block, int smem, cudaStream_t s, bool pdl,
                            int cl, const V&... args) {
  if (!pdl && cl == 1) {
    kernel<<<grid, block, smem, s>>>(args...);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  int na = 0;
  if (pdl) {
    at[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
  }
  if (cl > 1) {
    at[na].id = cudaLaunchAttributeClusterDimension;
    at[na].val.clusterDim.x = (unsigned)cl;
    at[na].val.clusterDim.y = 1;
    at[na].val.clusterDim.z = 1;
    ++na;
  }
  cfg.attrs = at;
  cfg.numAttrs = (unsigned)na;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <typename T, int N, int KIND, int R = default_rows<T, N>(), int PE = default_row_pe<T, N>(), int CL = 1,
          int CMP = 0>
static cudaError_t launch_row_kind(const DomainDev& d, cudaStream_t s) {
  using Geo = RowGeo<T, N, KIND, R, PE, CL, CMP>;
  static std::atomic<int> done{0};
  cudaError_t e = set_smem(row_kernel<T, N, KIND, R, PE, CL, CMP>, cmax(Geo::SMEM, kSpreadSmem), done);
  if (e != cudaSuccess) return e;
  Args<T> a = make_args<T>(d);
  CUtensorMap tm;
  memset(&tm, 0, sizeof(tm));
  constexpr int ri = R == 1 ? 0 : R == 2 ? 1 : R == 4 ? 2 : -1;
  if constexpr (Geo::TMA_OK && ri >= 0) {
    if (d.use_tma && d.tma_ok[ri] && d.err) {
      tm = d.tmapG[ri];
      a.tma = 1;
    }
  }
  const bool pdl = KIND == ROW_STEP && step_pdl<N>(d, s);
  return launch_k(row_kernel<T, N, KIND, R, PE, CL, CMP>, N / R, Geo::NT, launch_smem(Geo::SMEM, N / R, pdl ? spread_smem<T, N>(d) : 0), s, pdl,
                  CL, a, tm);
}

// (the other column modes take the first step variant's shape, so that a state read back and set
// again steps on bit for bit: the prologue makes the same row inputs as the step's column pass)
template <typename T, int N, int MODE, int PE = default_step_col_pe<T, N>()>
static cudaError_t launch_col_mode(const DomainDev& d, cudaStream_t s) {
  constexpr int LEAN = col_lean<T, N, MODE, PE>();
  using Geo = ColGeo<T, N, MODE, PE, LEAN>;
  static std::atomic<int> done{0};
  cudaError_t e = set_smem(col_kernel<T, N, MODE, PE, LEAN>, cmax(Geo::SMEM, kSpreadSmem), done);
  if (e != cudaSuccess) return e;
  // a recorded step adds one block that finishes the time-series sample
  const int extra = (MODE == COL_STEP && d.rec != nullptr) ? 1 : 0;
  const bool pdl = MODE == COL_STEP && step_pdl<N>(d, s);
  return launch_k(col_kernel<T, N, MODE, PE, LEAN>, Geo::H + extra, Geo::NT, launch_smem(Geo::SMEM, Geo::H + extra, pdl ? spread_smem<T, N>(d) : 0), s,
                  pdl, 1, make_args<T>(d));
}

template <typename T, int N, int KIND>
static cudaError_t launch_row_io(const DomainDev& d, cudaStream_t s) {
  constexpr int R = default_rows<T, N>(), PE = default_row_pe<T, N>();
  using Geo = RowGeo<T, N, KIND, R, PE>;
  static std::atomic<int> done{0};
  cudaError_t e = set_smem(row_io_kernel<T, N, KIND, R, PE>, Geo::SMEM, done);
  if (e != cudaSuccess) return e;
  row_io_kernel<T, N, KIND, R, PE><<<N / R, Geo::NT, Geo::SMEM, s>>>(make_args<T>(d), d.io);
  return cudaGetLastError();
}

template <typename T, int N>
static cudaError_t launch_row(int kind, const DomainDev& d, cudaStream_t s) {
  switch (kind) {
    case K_ROW_STEP: return launch_row_kind<T, N, ROW_STEP>(d, s);
    case K_ROW_FWD_VEL: return launch_row_kind<T, N, ROW_FWD_VEL>(d, s);
    case K_ROW_FWD_MASK: return launch_row_kind<T, N, ROW_FWD_MASK>(d, s);
    case K_ROW_INV_FIELDS: return launch_row_kind<T, N, ROW_INV_FIELDS>(d, s);
    case K_ROW_INV_MASK: return launch_row_kind<T, N, ROW_INV_MASK>(d, s);
    case K_ROW_INV_DIAG: return launch_row_kind<T, N, ROW_INV_DIAG>(d, s);
    case K_ROW_FEATURES: return launch_row_io<T, N, ROW_FEATURES>(d, s);
    case K_ROW_FWD_CORR: return launch_row_io<T, N, ROW_FWD_CORR>(d, s);
  }
  return cudaErrorInvalidValue;
}

template <typename T, int N>
static int row_blocks(int kind) {
  (void)kind;
  return N / default_rows<T, N>();
}

template <typename T, int N>
static cudaError_t launch_col(int mode, const DomainDev& d, cudaStream_t s) {
  switch (mode) {
    case K_COL_STEP: return launch_col_mode<T, N, COL_STEP>(d, s);
    case K_COL_PROLOGUE: return launch_col_mode<T, N, COL_PROLOGUE>(d, s);
    case K_COL_PROJECT: return launch_col_mode<T, N, COL_PROJECT>(d, s);
    case K_COL_MASK: return launch_col_mode<T, N, COL_MASK>(d, s);
    case K_COL_ADDW: return launch_col_mode<T, N, COL_ADDW>(d, s);
    case K_COL_DIV: return launch_col_mode<T, N, COL_DIV>(d, s);
  }
  return cudaErrorInvalidValue;
}

template <typename T, int N>
static cudaError_t launch_spec(const DomainDev& d, int nbins, cudaStream_t s) {
  constexpr int H = N / 4 + 1;
  spectrum_col_kernel<T, N><<<H, 256, 0, s>>>(make_args<T>(d), nbins, d.colhist, d.bad);
  return cudaGetLastError();
}

template <typename T, int N, int R, int PE>
static cudaError_t launch_row_batched(const void* args, int ndom, cudaStream_t s) {
  using Geo = RowGeo<T, N, ROW_STEP, R, PE>;
  row_kernel_batched<T, N, ROW_STEP, R, PE><<<dim3(N / R, ndom), Geo::NT, Geo::SMEM, s>>>(
      static_cast<const Args<T>*>(args));
  return cudaGetLastError();
}

template <typename T, int N, int R, int PE>
static cudaError_t prepare_row_batched() {
  static std::atomic<int> done{0};
  return set_smem(row_kernel_batched<T, N, ROW_STEP, R, PE>, RowGeo<T, N, ROW_STEP, R, PE>::SMEM, done);
}

template <typename T, int N, int PE>
static cudaError_t launch_col_batched(const void* args, int ndom, cudaStream_t s) {
  using Geo = ColGeo<T, N, COL_STEP, PE>;
  col_kernel_batched<T, N, COL_STEP, PE><<<dim3(Geo::H, ndom), Geo::NT, Geo::SMEM, s>>>(
      static_cast<const Args<T>*>(args));
  return cudaGetLastError();
}

template <typename T, int N, int PE>
static cudaError_t prepare_col_batched() {
  static std::atomic<int> done{0};
  return set_smem(col_kernel_batched<T, N, COL_STEP, PE>, ColGeo<T, N, COL_STEP, PE>::SMEM, done);
}

template <typename T>
static void pack_args(const DomainDev& d, void* dst) {
  const Args<T> a = make_args<T>(d);
  memcpy(dst, &a, sizeof(a));
}

// (again: a shape that is in the list already gets this index as well)
template <typename T, int N, int R, int PE, int CL = 1, int CMP = 0>
static void add_row_variant(SizeOps& o, bool again = false) {
  if constexpr (RowGeo<T, N, ROW_STEP, R, PE, CL, CMP>::VALID &&
                (N >= 64 || (R == default_step_rows<T, N>() && PE == default_step_row_pe<T, N>() && CL == 1 && CMP == 0))) {
    // a compact variant whose plan equals the plain one's (nothing to leave out) is the same shape
    constexpr int cmp =
        RowGeo<T, N, ROW_STEP, R, PE, CL, CMP>::SMEM != RowGeo<T, N, ROW_STEP, R, PE, CL, 0>::SMEM ? CMP : 0;
    for (int i = 0; i < o.n_row_variants && !again; ++i)
      if (o.row_step[i].rows == R && o.row_step[i].pe == cmin(PE, N / 2) && o.row_step[i].cl == CL &&
          o.row_step[i].cmp == cmp)
        return;   // same shape
    StepVariant v{&launch_row_kind<T, N, ROW_STEP, R, PE, CL, CMP>, nullptr, nullptr, R, cmin(PE, N / 2), CL, cmp,
                  RowGeo<T, N, ROW_STEP, R, PE, CL, CMP>::TMA_OK ? 1 : 0};
    if constexpr (N <= kMaxBatchN && CL == 1 && CMP == 0) {
      v.batched = &launch_row_batched<T, N, R, PE>;
      v.prepare = &prepare_row_batched<T, N, R, PE>;
    }
    if (o.n_row_variants < kMaxVariants) o.row_step[o.n_row_variants++] = v;
  }
}

template <typename T, int N, int PE>
static void add_col_variant(SizeOps& o, bool again = false) {
  if constexpr (ColGeo<T, N, COL_STEP, PE>::VALID && (N >= 64 || PE == default_step_col_pe<T, N>())) {
    for (int i = 0; i < o.n_col_variants && !again; ++i)
      if (o.col_step[i].pe == cmin(PE, N)) return;
    StepVariant v{&launch_col_mode<T, N, COL_STEP, PE>, nullptr, nullptr, 1, cmin(PE, N), 1, 0};
    if constexpr (N <= kMaxBatchN) {
      v.batched = &launch_col_batched<T, N, PE>;
      v.prepare = &prepare_col_batched<T, N, PE>;
    }
    if (o.n_col_variants < kMaxVariants) o.col_step[o.n_col_variants++] = v;
  }
}

// Index of the unclustered variant of this shape, 0 if there is none.
inline int find_shape(const StepVariant* v, int n, int rows, int pe, int cmp) {
  for (int i = 0; i < n; ++i)
    if (v[i].rows == rows && v[i].pe == pe && v[i].cl == 1 && v[i].cmp == cmp) return i;
  return 0;
}

template <typename T, int N>
static SizeOps make_ops() {
  SizeOps o;
  o.row = &launch_row<T, N>;
  o.col = &launch_col<T, N>;
  o.spec = &launch_spec<T, N>;
  o.row_blocks = &row_blocks<T, N>;
  o.n_row_variants = 0;
  o.n_col_variants = 0;
  o.args_bytes = (int)sizeof(Args<T>);
  o.pack_args = &pack_args<T>;
  add_row_variant<T, N, default_step_rows<T, N>(), default_step_row_pe<T, N>(), default_row_cluster<T, N>()>(o);
  if constexpr (sizeof(T) == 4 && N == 1024) add_col_variant<T, N, default_col_pe<T, N>()>(o);
  add_col_variant<T, N, default_step_col_pe<T, N>()>(o);
  if constexpr (sizeof(T) == 4) {
    add_row_variant<T, N, 4, 16>(o);
    add_row_variant<T, N, 2, 16>(o);
    add_row_variant<T, N, 1, 16>(o);
    add_row_variant<T, N, 2, 8>(o);
    if constexpr (N >= 2048) {
      // clusters of two blocks: global segments of 2R values (large grids, where R is small)
      add_row_variant<T, N, 1, 16, 2>(o);
      add_row_variant<T, N, 2, 16, 2>(o);
    }
    if constexpr (N >= 1024 && N <= 4096) {
      // compact: in-place forward transforms, mask rows not staged: two or more blocks per SM
      add_row_variant<T, N, 2, 16, 1, 1>(o);
      add_row_variant<T, N, 1, 16, 2, 1>(o);
      add_row_variant<T, N, 1, 16, 1, 1>(o);
    }
    add_col_variant<T, N, 8>(o);
    add_col_variant<T, N, 16>(o);
    add_col_variant<T, N, 4>(o);
  } else {
    // Up to 256^2 the default is one of the other shapes; those keep the indices by which saved plans
    // name them (rows 1: one row, 8 points; 2: one row, 4 points; columns 1: 4 points).
    if constexpr (N >= 64 && N <= 256) {
      add_row_variant<T, N, 1, 8>(o, true);
      add_row_variant<T, N, 1, 4>(o, true);
      add_col_variant<T, N, 4>(o, true);
    }
    add_row_variant<T, N, 2, 8>(o);
    add_row_variant<T, N, 1, 8>(o);
    add_row_variant<T, N, 1, 4>(o);
    add_col_variant<T, N, 8>(o);
    add_col_variant<T, N, 4>(o);
  }
  // One domain by itself leaves most of the GPU idle up to 256^2: small tiles then spread it over
  // more blocks and halve the butterflies of a thread's chain (float, us a step: 64^2 6.3 -> 4.9,
  // 256^2 7.3 -> 6.0; double 64^2 26 -> 17, 256^2 40 -> 35).
  constexpr bool F32 = sizeof(T) == 4;
  // The prologue that starts a call has the column step's shape: it rounds the row inputs as the step
  // it stands for would have, so that calls of k steps and one of 2k leave the same bits.  (Grids
  // below 64^2 have one column variant.)
  constexpr int ALONE_PE = N < 64 ? default_step_col_pe<T, N>() : F32 || N <= 256 ? 4 : 8;
  o.alone_row = find_shape(o.row_step, o.n_row_variants, F32 ? (N <= 256 ? 2 : 4) : (N <= 256 ? 1 : 2),
                           F32 ? (N <= 256 ? 8 : 16) : (N <= 256 ? 4 : 8), 0);
  o.alone_col = find_shape(o.col_step, o.n_col_variants, 1, cmin(ALONE_PE, N), 0);
  o.alone_prologue = nullptr;
  if constexpr (N <= kAloneMaxN) o.alone_prologue = &launch_col_mode<T, N, COL_PROLOGUE, ALONE_PE>;
  // 2048^2 and 4096^2 float start with the compact two-row pass (46.1 and 219.5 us; the plain ones
  // 57.0 and 232)
  o.start_row = F32 && (N == 2048 || N == 4096) ? find_shape(o.row_step, o.n_row_variants, 2, 16, 1) : 0;
  o.start_col = F32 && N == 1024 ? find_shape(o.col_step, o.n_col_variants, 1, default_step_col_pe<T, N>(), 0) : 0;
  return o;
}

bool TTSH_REGISTRY(int n, SizeOps* o) {
  switch (n) {
#define X(NN) \
  case NN: *o = make_ops<TTSH_T, NN>(); return true;
    TTSH_SIZES
#undef X
  }
  return false;
}

}  // namespace ttsh

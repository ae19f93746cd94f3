// Host-side index checks of the forms of the step kernels that tests/geometry_check.cu, whose
// checks these build on, does not go through:
//   - the band-limited transforms: the first stage loads exactly the elements inside the band,
//     each from the stored column, and the last stage stores every element read afterwards;
//   - the shared twiddle tables, cut to the entries the passes use;
//   - row bodies in place with staged mask rows (CMP = 2) and column bodies without a staging
//     area (LEAN = 1): the persistent stepper's shapes, and the column steps that take the
//     lean form;
//   - the row kinds that exchange fields with the corrector network, and the column modes in the
//     shape they are launched in;
//   - the real-space terms in place: every complex slot visited once, its mask values inside
//     the block's rows.
// No GPU is needed.
#define main geometry_check_main
#include "geometry_check.cu"
#undef main

#include "ttsh_persist.cuh"

// ------------------------------------------------------------------ band-limited transforms
// In a column transform of length L the band is |m| <= L / 4.
template <typename T, int L, int PE>
static void check_band(const char* who) {
  constexpr int M = L / 4, NK = 2 * M + 1;
  {   // first stage, inputs limited
    constexpr int R = stage_radix(L, PE, 1);
    CHECK(R >= 4, "%s: radix %d", who, R);
    const int SL = L / R;
    std::vector<int> rd(L, 0);
    for (int q = 0; q < SL; ++q)
      for (int r = 0; r < R; ++r) {
        if (r > R / 4 && r < 3 * R / 4) continue;
        if (r == R / 4 && q != 0) continue;
        const int idx = q + r * SL;
        const bool upper = r >= R / 2;
        CHECK(upper == (idx >= L / 2), "%s idx %d", who, idx);
        const int ky = upper ? idx - L : idx, j = upper ? idx - L + NK : idx;   // the functor's stored mode
        CHECK(ky >= -M && ky <= M && j >= 0 && j < NK && (j <= M ? j : j - NK) == ky, "%s idx %d j %d", who, idx, j);
        ++rd[idx];
      }
    for (int i = 0; i < L; ++i) CHECK(rd[i] == (i <= M || i >= L - M ? 1 : 0), "%s element %d", who, i);
  }
  {   // last stage, outputs limited
    int Ns = 1;
    while (Ns * stage_radix(L, PE, Ns) < L) Ns *= stage_radix(L, PE, Ns);
    const int R = stage_radix(L, PE, Ns);
    std::vector<int> wr(L, 0);
    for (int q = 0; q < L / R; ++q) {
      const int k = q & (Ns - 1), base = (q - k) * R + k;
      for (int r = 0; r < R; ++r)
        if (R < 4 || r <= R / 4 || r >= 3 * R / 4) ++wr[base + r * Ns];
    }
    for (int ky = -M; ky <= M; ++ky) CHECK(wr[ky & (L - 1)] == 1, "%s output %d", who, ky);
  }
}

// ------------------------------------------------------------------ twiddle tables
// An index into W_TWN through the table's levels stays inside the `entries` that were filled.
template <typename T, int TWN>
static void check_twiddle(const char* who, int m, int entries) {
  using TW = TwTab<T, TWN>;
  if (TW::NHI == 1) {
    CHECK(m >= 0 && m < entries && m < TW::NLO, "%s twiddle %d of %d", who, m, entries);
  } else {
    CHECK(m >= 0 && (m >> TW::SB) < TW::NHI && entries == TW::ENTRIES, "%s twiddle %d of %d", who, m, entries);
  }
}
template <typename T, int L, int PE, int TWN>
static void check_stage_twiddles(const char* who, int entries) {
  if constexpr (!StageTab<T, L, PE>::USE) {   // (else the stages have tables of their own)
    for (int Ns = 1; Ns < L; Ns *= stage_radix(L, PE, Ns)) {
      const int R = stage_radix(L, PE, Ns), stride = TWN / (Ns * R);
      if (Ns > 1)
        for (int r = 1; r < R; ++r) check_twiddle<T, TWN>(who, r * (Ns - 1) * stride, entries);
    }
  }
}

// ------------------------------------------------------------------ row pass
template <typename T, int N, int KIND, int R, int PEV, int CL = 1, int CMP = 0>
static void check_row_form() {
  using G = RowGeo<T, N, KIND, R, PEV, CL, CMP>;
  if constexpr (G::VALID) {
    check_row<T, N, KIND, R, PEV, CL, CMP>();
    char who[96];
    std::snprintf(who, sizeof who, "row form %s N=%d kind=%d R=%d PE=%d CL=%d CMP=%d", tname<T>(), N, KIND, R, PEV, CL, CMP);
    CHECK(G::NT % 32 == 0 && G::NT <= 1024, "%s", who);   // named barriers count whole warps
    constexpr int kStageBytes = StageTab<T, G::L, G::PE>::BYTES;
    CHECK(G::OFF_STAB >= G::TW_ENT * G::CB && G::TW_BYTES >= G::OFF_STAB + kStageBytes, "%s", who);
    check_stage_twiddles<T, G::L, G::PE, N>(who, G::TW_ENT);
    for (int k = 0; k < G::L; ++k) check_twiddle<T, N>(who, k, G::TW_ENT);   // the real-transform passes
    // element k of the inverse transform comes from one stored column
    for (int k = 0; k < G::L; ++k) {
      const int kk = k >= G::L / 2 ? G::L - k : k;
      CHECK(kk >= 0 && kk <= G::M, "%s element %d", who, k);
    }
    if (KIND == ROW_STEP && !G::SEPARATE) {   // the terms in place, KI complex slots a thread
      const int KI = (R * G::L + G::NT - 1) / G::NT;
      std::vector<int> seen(R * G::L, 0);
      for (int t = 0; t < G::NT; ++t)
        for (int i = 0; i < KI; ++i) {
          const int e = t + i * G::NT;
          if (e >= R * G::L) break;
          ++seen[e];
          CHECK(((e / G::L) + 2 * R) * G::LPR + padded(e % G::L, G::PS) < G::BUF_BYTES / G::CB, "%s slot %d", who, e);
          CHECK(2 * e + 1 < R * N, "%s mask %d", who, e);   // two mask values of the block's R rows
        }
      for (int e = 0; e < R * G::L; ++e) CHECK(seen[e] == 1, "%s slot %d", who, e);
    }
  }
}

// ------------------------------------------------------------------ column pass
template <typename T, int N, int MODE, int PEV, int LEAN = 0>
static void check_col_form() {
  using G = ColGeo<T, N, MODE, PEV, LEAN>;
  if constexpr (G::VALID) {
    ++g_checked;
    char who[96];
    std::snprintf(who, sizeof who, "col form %s N=%d mode=%d PE=%d LEAN=%d", tname<T>(), N, MODE, PEV, LEAN);
    constexpr int CB = G::CB, LP = G::LP, PS = G::PS;
    check_fft<T, N, G::PE>(who);
    check_band<T, N, G::PE>(who);
    CHECK(G::NT % 32 == 0 && G::NT % G::TT == 0 && G::FB >= 1, "%s", who);
    CHECK(LEAN == 0 || !G::BULK, "%s", who);
    constexpr int kStageBytes = StageTab<T, N, G::PE>::BYTES;
    CHECK(G::OFF_STAB >= G::TW_ENT * CB && G::TW_BYTES >= G::OFF_STAB + kStageBytes, "%s", who);
    check_stage_twiddles<T, N, G::PE, N>(who, G::TW_ENT);
    CHECK(G::OFF_BUF >= G::TW_BYTES && G::OFF_BUF % 16 == 0, "%s", who);
    CHECK(G::OFF_ACC % 16 == 0 && G::OFF_ACC >= G::OFF_BUF + G::FB * LP * CB, "%s", who);
    CHECK(G::OFF_WS % 16 == 0 && G::OFF_WS >= G::OFF_ACC + G::NK * CB, "%s", who);
    CHECK(G::OFF_STG % 16 == 0 && G::OFF_STG >= G::OFF_WS + (G::WS_BYTES > 0 ? G::NK * CB : 0), "%s", who);
    CHECK(G::OFF_S0 % 16 == 0 && G::OFF_S0 >= G::OFF_STG + (G::BULK ? G::NF * N * CB : 0), "%s", who);
    CHECK(G::SMEM >= G::OFF_S0 + 4 * (int)sizeof(T), "%s", who);
    CHECK(cmax(G::SMEM, kSpreadSmemBytes) + kRecSmem <= 227 * 1024, "%s launch bytes", who);
    // columns staged into the transform buffers (no staging area)
    for (int b = 0; b < G::FB; ++b)
      for (int y = 0; y < N; ++y) CHECK(b * LP + padded(y, PS) < G::FB * LP, "%s buf b=%d y=%d", who, b, y);
    // bulk copies go to a multiple of 16 bytes, whole units
    if (G::BULK) CHECK((N * CB) % 16 == 0, "%s", who);
  }
}

template <typename T, int N, int PE>
static void check_col_step() {
  if constexpr (ColGeo<T, N, COL_STEP, PE>::VALID) check_col_form<T, N, COL_STEP, PE, col_lean<T, N, COL_STEP, PE>()>();
}

// ------------------------------------------------------------------ the persistent stepper
template <typename T, int N, bool LF>
static void check_persist() {
  using S = PersistShape<T, N, LF>;
  using P = PersistLimits<T, LF>;
  check_row_form<T, N, ROW_STEP, S::R, S::RPE, 1, S::CMP>();
  check_col_form<T, N, COL_STEP, S::CPE, S::LEAN>();
  CHECK(S::RG::VALID && S::CG::VALID, "persistent N=%d", N);
  CHECK(S::RG::SMEM <= P::SMEM && S::CG::SMEM <= P::SMEM && S::RG::NT <= P::NT && S::CG::NT <= P::NT, "persistent N=%d", N);
}

template <typename T, int N>
static void check_forms() {
  check_row_form<T, N, ROW_STEP, default_step_rows<T, N>(), default_step_row_pe<T, N>(), default_row_cluster<T, N>()>();
  check_row_form<T, N, ROW_STEP, 4, 16>();
  check_row_form<T, N, ROW_STEP, 2, 16>();
  check_row_form<T, N, ROW_STEP, 1, 16>();
  check_row_form<T, N, ROW_STEP, 2, 8>();
  check_row_form<T, N, ROW_STEP, 1, 8>();
  check_row_form<T, N, ROW_STEP, 1, 4>();
  if constexpr (sizeof(T) == 4 && N >= 2048) {
    check_row_form<T, N, ROW_STEP, 1, 16, 2>();
    check_row_form<T, N, ROW_STEP, 2, 16, 2>();
  }
  if constexpr (sizeof(T) == 4 && N >= 1024 && N <= 4096) {
    check_row_form<T, N, ROW_STEP, 2, 16, 1, 1>();
    check_row_form<T, N, ROW_STEP, 1, 16, 2, 1>();
    check_row_form<T, N, ROW_STEP, 1, 16, 1, 1>();
  }
  constexpr int R = default_rows<T, N>(), RPE = default_row_pe<T, N>();
  check_row_form<T, N, ROW_INV_FIELDS, R, RPE>();
  check_row_form<T, N, ROW_INV_DIAG, R, RPE>();
  check_row_form<T, N, ROW_FWD_VEL, R, RPE>();
  check_row_form<T, N, ROW_FWD_MASK, R, RPE>();
  check_row_form<T, N, ROW_INV_MASK, R, RPE>();
  check_row_form<T, N, ROW_FEATURES, R, RPE>();
  check_row_form<T, N, ROW_FWD_CORR, R, RPE>();
  check_col_step<T, N, 16>();
  check_col_step<T, N, 8>();
  check_col_step<T, N, 4>();
  // the other modes in the shape of the step's default, the prologue also in the others
  constexpr int CPE = default_step_col_pe<T, N>();
  check_col_form<T, N, COL_PROLOGUE, CPE>();
  check_col_form<T, N, COL_PROJECT, CPE>();
  check_col_form<T, N, COL_MASK, CPE>();
  check_col_form<T, N, COL_ADDW, CPE>();
  check_col_form<T, N, COL_DIV, CPE>();
  check_col_form<T, N, COL_PROLOGUE, 8>();
  check_col_form<T, N, COL_PROLOGUE, 4>();
  if constexpr (N <= kPersistMaxN) {
    check_persist<T, N, false>();
    check_persist<T, N, sizeof(T) == 4>();
  }
}

// The persistent kernel's blocks, as many as it is compiled for, fit an SM.
template <typename T, bool LF>
static void check_persist_residency() {
  using P = PersistLimits<T, LF>;
  CHECK((P::SMEM + 128 + 1024 + 512) * persist_blocks<T>(LF) <= 228 * 1024, "persistent blocks %d", P::SMEM);
  CHECK((P::NT + 32) * persist_blocks<T>(LF) <= 2048, "persistent threads %d", P::NT);
}

int main() {
  check_forms<float, 16>();
  check_forms<float, 32>();
  check_forms<float, 64>();
  check_forms<float, 128>();
  check_forms<float, 256>();
  check_forms<float, 512>();
  check_forms<float, 1024>();
  check_forms<float, 2048>();
  check_forms<float, 4096>();
  check_forms<float, 8192>();
  check_forms<double, 16>();
  check_forms<double, 32>();
  check_forms<double, 64>();
  check_forms<double, 128>();
  check_forms<double, 256>();
  check_forms<double, 512>();
  check_forms<double, 1024>();
  check_forms<double, 2048>();
  check_forms<double, 4096>();
  check_persist_residency<float, false>();
  check_persist_residency<float, true>();
  check_persist_residency<double, false>();
  std::printf("%d pass forms checked, %d failures\n", g_checked, g_fail);
  return g_fail == 0 && g_checked > 0 ? 0 : 1;
}

// Host checks of which kernel, form and stream a call takes, on layout-only
// plans (no GPU): one check per name on the command line.
#include "capi.cu"

// Host allocations, counted.
static size_t allocations = 0;
void* operator new(size_t n) {
#ifndef __CUDA_ARCH__
  ++allocations;
#endif
  return malloc(n ? n : 1);
}
void operator delete(void* p) noexcept { free(p); }
void operator delete(void* p, size_t) noexcept { free(p); }

namespace {

int failures = 0;
void expect(bool ok, const char* what) {
  if (!ok) {
    std::printf("FAILED: %s\n", what);
    ++failures;
  }
}

// The kernels of the direct form are compiled for its own fields.
void direct_gemm() {
  NbrGemm g{};
  const DirectGemm& d = g;
  expect(sizeof(DirectGemm) < sizeof(NbrGemm), "the direct form's description holds its own fields only");
  expect(reinterpret_cast<const char*>(&d) == reinterpret_cast<const char*>(&g), "its fields come first");
}

// A plan's layout without device memory, with placeholder side streams.
struct Dry {
  fmm_plan_t P;
  Dry(int nx, int ny, int nz, int order, int leaf, const fmm_opts& o) : P(new fmm_plan_s) {
    P->static_base = reinterpret_cast<unsigned char*>((uintptr_t)1 << 40);
    P->static_cap = (size_t)1 << 39;
    P->static_keep_tables = P->dry = true;
    const int d3[3] = {nx, ny, nz};
    expect(plan_init(P, d3, 1.0, 1.0, order, leaf, o, nullptr, 0) == FMM_OK, fmm_last_error());
  }
  ~Dry() { delete P; }
};
fmm_opts opts(int precision, int accel, int final_stage = 0) {
  fmm_opts o;
  fmm_default_opts(&o);
  o.precision = precision;
  o.accel = accel;
  o.final_stage = final_stage;
  return o;
}

// The levels beside a leaf-8 near field off the tensor cores run at its own
// priority; with the final-stage M2P on the high-priority stream, a split near
// field behind it.  The transpose of the analytic force at leaf 4: ahead of
// the near field on the caller's stream (FP32: order 5 on, 17 to 152 blocks).
void leaf8_streams() {
  cudaStream_t hi = reinterpret_cast<cudaStream_t>(16), lo = reinterpret_cast<cudaStream_t>(32);
  cudaStream_t own = reinterpret_cast<cudaStream_t>(48);
  for (int leaf : {2, 4, 8})
    for (int prec : {FMM_FP32, FMM_FP64})
      for (int m2p : {0, 1}) {
        Dry d(leaf * 12, leaf * 12, leaf * 12, 4, leaf, opts(prec, 1, m2p));
        d.P->side = hi, d.P->side2 = lo;
        const bool flat = leaf == 8 && !m2p;
        expect(levels_stream(d.P, false, own) == (flat ? lo : hi), "levels' stream of a forward solve");
        // the transposed force's near field: 12 tiles (2 x 3 x 2) times its column tiles
        for (int order : {4, 5, 8})
          for (int nt : {1, 2, 12, 13}) {
            d.P->p = order;
            d.P->near_adj_ntiles = nt;
            const bool ahead = leaf == 4 && !m2p && (prec == FMM_FP64 || (order >= 5 && (nt == 2 || nt == 12)));
            expect(levels_stream(d.P, true, own) == (ahead ? own : hi), "levels' stream of the transposed force");
          }
        for (int split : {1, 3}) {
          d.P->near_choice.dsplit = split;
          expect(near_behind(d.P, false, false) == (leaf == 8 && m2p && split > 1), "near field behind the final stage");
          expect(near_behind(d.P, false, true) == (split > 1), "a split near field beside a tensor-core level");
          expect(!near_behind(d.P, true, false) && !near_behind(d.P, true, true),
                 "the transposed force's near field is unsplit");
        }
        d.P->side = d.P->side2 = nullptr;
      }
}

// Fused FP32 batches: with leaf-8 fields one wide direct launch per tile shape
// (their leaf level included); other leaves run it in the reflection basis.
void leaf8_batch() {
  for (std::array<int, 2> leaf : {std::array<int, 2>{4, 4}, {8, 8}, {4, 8}, {2, 2}}) {
    Dry a(leaf[0] * 8, leaf[0] * 12, leaf[0] * 12, 4, leaf[0], opts(FMM_FP32, 1));
    Dry b(leaf[1] * 12, leaf[1] * 10, leaf[1] * 24, 4, leaf[1], opts(FMM_FP32, 1));
    fmm_batch_s B;
    B.plans = {a.P, b.P};
    build_fused<float>(&B, nullptr, nullptr, nullptr, true);
    int sym = 0, gemm = 0;
    for (const MultiStep& st : B.steps) {
      if (st.kind != MK_GEMM) continue;
      ++gemm;
      sym += st.kn[0] + st.kn[1];
      expect(st.wide == (leaf[0] == 8 || leaf[1] == 8), "wide form with leaf-8 fields");
    }
    const int want = (leaf[0] == 4 ? 2 : leaf[0] == 2 ? 1 : 0) + (leaf[1] == 4 ? 2 : leaf[1] == 2 ? 1 : 0);
    expect(gemm > 0 && sym == want, "reflection-basis items (leaf level, near field of leaf 4)");
  }
}

// The far field's launches: the FP64 levels of a mixed plan, the row groups, the
// narrow group, the other levels; every level once, without a host allocation.
void far_order() {
  auto kinds = [](fmm_plan_t P) {
    int ls[kMaxLevels], n = 0, seen = 0;
    for (int l = 2; l <= P->L; ++l)
      if (!P->lev[l].tc && !(l == P->L && P->m2p)) ls[n++] = l;
    FarItem items[kMaxLevels];
    const size_t before = allocations;
    const int m = far_items(P, ls, n, items);
    (void)fmm_solve_launches(P, 1);
    expect(allocations == before, "no host allocation (an exception would cross the C interface)");
    std::string s;
    bool once[kMaxLevels] = {};
    for (int i = 0; i < m; ++i) {
      s += items[i].kind == FarItem::kRows ? 'r' : items[i].kind == FarItem::kNarrow ? 'n' : 'l';
      for (int k = 0; k < items[i].n; ++k) {
        expect(!once[items[i].ls[k]], "a level once");
        once[items[i].ls[k]] = true;
        ++seen;
      }
    }
    expect(seen == n, "every level");
    return s;
  };
  Dry fp32(64, 64, 64, 6, 4, opts(FMM_FP32, 1));
  expect(kinds(fp32.P) == "r", "levels of at most 512 rows in one group");
  Dry mid(96, 96, 96, 6, 4, opts(FMM_FP32, 1));
  expect(kinds(mid.P) == "rl", "the group ahead of the leaf level");
  // Cartesian: the unsplit leaf level in the narrow form ahead of the split one above it
  fmm_opts o = opts(FMM_FP32, 1);
  o.m2l_cartesian = 1;
  Dry cart(160, 160, 160, 6, 4, o);
  expect(cart.P->m2l_choice[5].dsplit > 1 && narrow_level(cart.P, 6) && kinds(cart.P) == "rnl", "the narrow group second");
  // the levels of a mixed plan with FP64 coarse levels: two of those (one column
  // per lane, split), then FP32 ones in row groups
  Dry mixed(128, 128, 128, 0, 4, opts(FMM_FP32, 1));
  mixed.P->tc_kind = TC_BF16X3;
  for (int l : {2, 3}) mixed.P->lev[l].f64 = 1, mixed.P->m2l_choice[l].shape = 3;
  for (int l = 2; l <= mixed.P->L; ++l) mixed.P->m2l_choice[l].dsplit = 27;
  for (int l = 4; l <= mixed.P->L; ++l) mixed.P->m2l_choice[l].shape = 0;
  expect(kinds(mixed.P).substr(0, 3) == "llr", "the FP64 levels ahead of the row groups");
}

// The near field's own scratch takes every split that the M2L's, which it used
// to share, held: 64 MiB or what a split M2L level needs.
void near_scratch() {
  struct {
    int n[3], order, precision;
  } cases[] = {{{96, 96, 64}, 6, FMM_FP64}, {{96, 96, 64}, 7, FMM_FP64}, {{64, 64, 64}, 6, FMM_FP64},
               {{96, 112, 128}, 4, FMM_FP32}, {{32, 40, 24}, 3, FMM_FP32}};
  for (const auto& c : cases) {
    Dry d(c.n[0], c.n[1], c.n[2], c.order, 4, opts(c.precision, 1));
    const size_t es = d.P->esize(), one = (size_t)d.P->ncell() * es;
    const NbrGemm g = near_gemm(d.P);
    for (int split : {27, 9, 3})
      if (split * one <= std::max(d.P->part_cap, (size_t)64 << 20))
        expect(choice_valid(d.P, g, d.P->h_near_tile_k, es, {split == 27 ? 0 : 1, split}), "a near-field split that fits");
    expect(d.P->near_part_off >= d.P->part_off + d.P->part_cap &&
               d.P->near_part_off + d.P->near_part_cap <= d.P->arena_bytes, "scratch of its own, inside the arena");
  }
}

// A level of a tensor-core precision that runs on the CUDA cores says so, and
// its variant can be read but not set.
void level_kind() {
  Dry d(64, 64, 64, 4, 4, opts(FMM_FP32, 0));
  Level& lv = d.P->lev[d.P->L];
  lv.tc = 1;
  lv.rfold_off = lv.fold_off, lv.rred_off = lv.lred_off;
  lv.fold_off = lv.lred_off = 0;
  int shape = -1, split = -1;
  expect(fmm_plan_level_kind(d.P, d.P->L) == 1, "kind of a small bf16x3 level: FP32 on the CUDA cores");
  expect(fmm_plan_tuning(d.P, d.P->L, &shape, &split) == FMM_OK && shape == d.P->m2l_choice[d.P->L].shape,
         "its variant reads");
  expect(fmm_plan_set_tuning(d.P, d.P->L, 1, 1) == FMM_ERR_ARG, "and stays as it is");
  d.P->use_refl = false;
  expect(fmm_plan_level_kind(d.P, d.P->L) == 3, "with a schedule selected: the tensor cores");
  expect(fmm_plan_tuning(d.P, d.P->L, &shape, &split) == FMM_ERR_ARG, "which have no variant");
  expect(fmm_plan_level_kind(d.P, 2) == 1, "an FP32 level");
}

// Prints 1 or 0 per contraction of a one-field fused batch, levels 2 to the
// leaf level and the near field: reflection basis or direct.
void batch_forms(int n, int order, int leaf, bool f64) {
  Dry d(n, n, n, order, leaf, opts(f64 ? FMM_FP64 : FMM_FP32, 1));
  fmm_batch_s B;
  B.plans = {d.P};
  if (f64)
    build_fused<double>(&B, nullptr, nullptr, nullptr, false);
  else
    build_fused<float>(&B, nullptr, nullptr, nullptr, false);
  std::vector<int> form(d.P->L, -1);  // level l at l - 2, the near field last
  for (const MultiStep& st : B.steps) {
    if (st.kind != MK_GEMM) continue;
    const NbrGemm* g = reinterpret_cast<const NbrGemm*>(B.h_tab.data() + st.args_off);
    for (int i = 0; i < st.n; ++i) {
      const bool near = !g[i].skip_center;
      int l = d.P->L;
      while (!near && (long long)g[i].grid[0] * g[i].grid[1] * g[i].grid[2] != d.P->lev[l].npar) --l;
      form[near ? d.P->L - 1 : l - 2] = i < st.kn[0] + st.kn[1];
    }
  }
  for (int v : form) {
    expect(v >= 0, "every contraction once");
    std::printf("%d ", v);
  }
}

}  // namespace

int main(int argc, char** argv) {
  const std::string what = argc > 1 ? argv[1] : "";
  if (what == "direct_gemm") direct_gemm();
  else if (what == "leaf8_streams") leaf8_streams();
  else if (what == "leaf8_batch") leaf8_batch();
  else if (what == "far_order") far_order();
  else if (what == "near_scratch") near_scratch();
  else if (what == "level_kind") level_kind();
  else if (what == "batch_forms" && argc == 6) batch_forms(atoi(argv[2]), atoi(argv[3]), atoi(argv[4]), atoi(argv[5]) != 0);
  else expect(false, "unknown check");
  return failures ? 1 : 0;
}

// Host checks of which kernel, form and stream a call takes, on layout-only
// plans (no GPU): one check per name on the command line.
#include "capi.cu"

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

}  // namespace

int main(int argc, char** argv) {
  const std::string what = argc > 1 ? argv[1] : "";
  if (what == "direct_gemm") direct_gemm();
  else expect(false, "unknown check");
  return failures ? 1 : 0;
}

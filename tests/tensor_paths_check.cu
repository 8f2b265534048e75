// Tensor generation with and without memory for its radial tables: the stored
// octant, in FP64 and in FP32, must be the same bytes (a user's plan has room
// for both tables, a serving plan only for that of U^eps).  Prints one line per
// grid and differing path, then "grids N differing D".
#include <cstdio>
#include <cstring>
#include <vector>

#include "../paper_2504_19410_gb300/csrc/fsa_internal.h"

namespace {
struct Case {
  fsa_kernel kernel;
  int n[3];
  double L[3], eps, param;
};
bool ok(cudaError_t e, const char* what) {
  if (e != cudaSuccess) std::printf("%s: %s\n", what, cudaGetErrorString(e));
  return e == cudaSuccess;
}
}  // namespace

int main() {
  const Case cases[] = {
      {FSA_KERNEL_COULOMB3D, {96, 96, 96}, {12, 12, 12}, 1.0, 0},       // cube: U and W radial
      {FSA_KERNEL_COULOMB3D, {192, 192, 192}, {16.1, 16.1, 16.1}, 0.7, 0},
      {FSA_KERNEL_COULOMB3D, {24, 48, 96}, {1.55, 3.1, 6.2}, 0.3, 0},   // one mesh step
      {FSA_KERNEL_COULOMB3D, {64, 64, 128}, {4, 4, 4}, 0.3, 0},         // one box
      {FSA_KERNEL_COULOMB3D, {128, 128, 128}, {8, 8, 12}, 0.5, 0},      // both in halves of the smallest step
      {FSA_KERNEL_COULOMB3D, {32, 24, 16}, {1.3, 1.7, 2.9}, 0.3, 0},    // no common ratio
      {FSA_KERNEL_BIHARMONIC3D, {64, 64, 64}, {4, 4, 4}, 0.3, 0},
      {FSA_KERNEL_YUKAWA3D, {48, 48, 48}, {3, 3, 3}, 0.4, 0.8},
  };
  int grids = 0, differing = 0;
  for (const Case& c : cases) {
    // a plan prepares the device for the grid's lengths
    fsa_plan_opts o{};
    o.eps = c.eps;
    o.eps_tol = -1.0;
    o.device = -1;
    o.kernel_param = c.param;
    fsa_plan* plan = nullptr;
    if (fsa_plan_create(&plan, c.kernel, 3, c.L, c.n, FSA_F64, &o) != FSA_OK) {
      std::printf("plan: %s\n", fsa_last_error());
      return 2;
    }
    const size_t total = (size_t)(c.n[0] + 1) * (c.n[1] + 1) * (c.n[2] + 1);
    double *oct = nullptr, *out = nullptr, *ut = nullptr, *wt = nullptr;
    if (!ok(cudaMalloc(&oct, total * 8), "oct") || !ok(cudaMalloc(&out, total * 8), "out") ||
        !ok(cudaMalloc(&ut, total / 4 * 8), "ut") || !ok(cudaMalloc(&wt, total / 4 * 8), "wt"))
      return 2;
    ++grids;
    bool same = true;
    for (const fsa_dtype dt : {FSA_F64, FSA_F32}) {
      const size_t bytes = total * (dt == FSA_F64 ? 8 : 4);
      std::vector<unsigned char> want(bytes), got(bytes);
      for (int mem = 3; mem >= 0; --mem) {
        if (!ok(cudaMemset(out, 0xff, bytes), "memset") ||
            !ok(fsa::tensorgen_run(c.kernel, c.n, c.L, c.eps, c.param, oct, out, dt, 0, nullptr, 0, mem & 1 ? ut : nullptr,
                                   mem & 2 ? wt : nullptr),
                "generate") ||
            !ok(cudaMemcpy(mem == 3 ? want.data() : got.data(), out, bytes, cudaMemcpyDeviceToHost), "copy"))
          return 2;
        if (mem < 3 && std::memcmp(want.data(), got.data(), bytes) != 0) {
          same = false;
          size_t k = 0;
          for (size_t i = 0; i < total; ++i) k += std::memcmp(&want[i * (bytes / total)], &got[i * (bytes / total)], bytes / total) != 0;
          std::printf("%dx%dx%d dtype %d: %s U table, %s W table: %zu of %zu points differ\n", c.n[0], c.n[1], c.n[2],
                      (int)dt, mem & 1 ? "with" : "no", mem & 2 ? "with" : "no", k, total);
        }
      }
    }
    differing += !same;
    cudaFree(oct);
    cudaFree(out);
    cudaFree(ut);
    cudaFree(wt);
    fsa_plan_destroy(plan);
  }
  std::printf("grids %d differing %d\n", grids, differing);
  return 0;
}

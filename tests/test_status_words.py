"""A bounded wait that expires in the tensor-core grouped GEMM is reported: its status word is among
those that a check reads and resets. The test program is the engine's host side with its internals in
reach, linked with the library's other objects."""

import pytest

from helpers import native_program, run_program

PROGRAM = r"""
#include "api.cu"
#include <cstdio>
#define EXPECT(c) do { if (!(c)) { printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)

int host() {
  int word = 0;
  int* dev[8];
  for (int n = 0; n < 4; ++n) {
    lipz_grid g{};
    g.bf = n & 1;
    g.dcgan = n >> 1;
    g.gemm_err = g.bf ? &word : nullptr;
    EXPECT(gemm_error_flag(&g) == g.gemm_err);
    flag_ptrs(&g, dev);
    int found = 0;
    for (int i = 0; i < 7; ++i) found += dev[i] == &word;
    EXPECT(found == (g.bf ? 1 : 0));
  }
  return 0;
}

// every kind of grid that runs the grouped GEMM: widths that the chained kernels do not take, a
// backward that they do not take (z = 128), and DCGANs with and without the tensor-core engine
int device() {
  for (int n = 0; n < 4; ++n) {
    lipz_arch a;
    EXPECT(lipz_arch_default(&a) == LIPZ_OK);
    a.precision = LIPZ_BF16;
    a.batch = 4;
    if (n == 0) a.hidden = 40;
    if (n == 1) a.z_dim = 128;
    if (n >= 2) {
      a.kind = LIPZ_DCGAN64;
      a.x_dim = 12288;
      a.z_dim = 100;
      a.ngf = a.ndf = n == 2 ? 32 : 64;
      a.mixture = 1;
    }
    lipz_grid* g = nullptr;
    EXPECT(lipz_grid_create(1, 1, &a, 5, &g) == LIPZ_OK);
    std::vector<float> pool((size_t)8 * a.x_dim, 0.25f);
    EXPECT(lipz_set_data(g, pool.data(), 8, a.x_dim) == LIPZ_OK);
    int* word = gemm_error_flag(g);
    EXPECT(word != nullptr);
    float fit[5];
    const int code = 2;
    EXPECT(lipz_eval_neighborhoods(g, fit, nullptr, nullptr, nullptr) == LIPZ_OK);
    EXPECT(cudaMemcpy(word, &code, 4, cudaMemcpyHostToDevice) == cudaSuccess);
    EXPECT(lipz_synchronize(g) == LIPZ_ERR_TIMEOUT);
    EXPECT(lipz_synchronize(g) == LIPZ_OK);
    EXPECT(cudaMemcpy(word, &code, 4, cudaMemcpyHostToDevice) == cudaSuccess);
    EXPECT(lipz_eval_neighborhoods(g, fit, nullptr, nullptr, nullptr) == LIPZ_ERR_TIMEOUT);
    EXPECT(lipz_eval_neighborhoods(g, fit, nullptr, nullptr, nullptr) == LIPZ_OK);
    EXPECT(lipz_grid_destroy(g) == LIPZ_OK);
  }
  return 0;
}

int main(int argc, char**) { return argc > 1 ? device() : host(); }
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    return native_program(tmp_path_factory, "status", PROGRAM, replaces=("api.cu",))


def test_every_status_word_is_listed(program):
    run_program(program)


@pytest.mark.gpu
def test_a_raised_word_is_reported_and_reset(program):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    run_program(program, "device")

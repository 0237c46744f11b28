"""The tensor-core grouped GEMM (bf16 networks that the chained kernels do not take): widths and
batches at the edges of its 128 x 64 and 128 x 128 tiles, of the 64-wide chunks and of the last MMA
step of 16, rows whose starts allow copies of 16, 8, 4 and 2 bytes, both operand orders (the
backward's transposed products), later minibatch steps, and the stored Gram matrix of a batch that is
too long for the Gram kernel; against the oracle, or the CUDA-core kernels. And the products' own
error, for every length of sum that the kernel takes."""

import numpy as np
import pytest

from helpers import native_program, run_program
from test_gpu_parity import L, _grid, _one_iteration_check, _pool  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols,batch,z,hidden,x", [
    (1, 1, 1, 1, 1, 1), (1, 2, 3, 5, 17, 33), (1, 2, 21, 16, 64, 63), (2, 2, 22, 50, 66, 130),
    (1, 3, 64, 15, 128, 65), (1, 2, 43, 100, 129, 127), (2, 3, 37, 48, 200, 500),
    (3, 3, 130, 66, 300, 1000), (4, 5, 24, 36, 257, 196), (1, 2, 65, 20, 512, 64)])
def test_one_iteration_against_the_oracle(L, rows, cols, batch, z, hidden, x):  # noqa: F811
    """Evaluation, gradients, Adam and weights by the rules of the one-iteration checks. (Nine cells
    at the largest size: the rules bound the median cell, and one cell with an activation that rounds
    the other way than the oracle's is off by 0.8 to 1.2 times 1e-2 on either route.)"""
    pool = _pool(7, 400, x)
    g = _grid(L, rows, cols, 29, pool, precision="bf16", batch=batch, z_dim=z, hidden=hidden,
              x_dim=x, keep_grads=1)
    _one_iteration_check(L, g, pool, 2e-2, label="bf16 h=%d" % hidden)


@pytest.mark.parametrize("batch,hidden,x,steps", [(30, 40, 50, 3), (1400, 24, 72, 1)])
def test_equals_the_cuda_core_kernels(L, batch, hidden, x, steps):  # noqa: F811
    """An iteration (several minibatch steps; a mixture on a stored Gram matrix) and the next
    evaluation on both routes. The fp32 sums differ in their order only, which moves a bf16 activation
    by at most one unit in the last place (2^-8); fitnesses and block means are means over many."""
    out = []
    for simt in (0, 1):
        g = L.Grid(1, 2, seed=3, precision="bf16", batch=batch, z_dim=10, hidden=hidden, x_dim=x,
                   train_steps=steps, mixture=1, force_simt=simt)
        g.set_data(_pool(4, 500, x))
        g.iterate(1)
        ev = g.eval()
        out.append((ev["fG"], ev["fD"], g.mixture(blocks=True)[1]))
        g.close()
    for a, b in zip(*out):
        assert np.max(np.abs(a - b)) <= 2.0 ** -7 * np.max(np.abs(b))


PROGRAM = r"""
#include "gemm_tc.cu"
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>
using namespace lipz;

// root mean square error against 64 bits of one 128 x 128 product over K: k_gemm_tc, and a chain of
// fp32 multiply-adds
int main() {
  std::mt19937 rng(1);
  std::normal_distribution<float> nd;
  constexpr int M = 128, N = 128, MAXK = 1024;
  const int lengths[10] = {GEMM_TC_MIN_K, GEMM_TC_MIN_K_STORE, 65, 80, 100, 128, GEMM_TC_CHUNK_K - 1,
                           GEMM_TC_CHUNK_K, 784, MAXK};
  bf16 *dA, *dB;
  float* dC;
  int* err;
  GemmDesc* dd;
  int2* dt;
  if (cudaMalloc(&dA, M * MAXK * 2) || cudaMalloc(&dB, N * MAXK * 2) || cudaMalloc(&dC, M * N * 4) ||
      cudaMalloc(&err, 4) || cudaMalloc(&dd, sizeof(GemmDesc)) || cudaMalloc(&dt, sizeof(int2)) ||
      cudaMemset(err, 0, 4) || cudaMemset(dt, 0, sizeof(int2)))
    return 1;
  for (int i = 0; i < 20; ++i) {
    const int K = lengths[i / 2];
    // operands as they come in a forward product, and in a weight gradient: deltas and activations
    // that are half zeros
    if (i % 2 && K < GEMM_TC_MIN_K_STORE) continue;
    auto value = [&] { return i % 2 && nd(rng) < 0 ? 0.f : nd(rng); };
    std::vector<bf16> A(M * K), B(N * K);
    for (bf16& x : A) x = __float2bfloat16(value());
    for (bf16& x : B) x = __float2bfloat16(i % 2 ? fabsf(value()) : value());
    GemmDesc d{};
    d.A = dA;
    d.B = dB;
    d.C = dC;
    d.sam = d.sbn = K;
    d.sak = d.sbk = d.scn = 1;
    d.scm = N;
    d.M = M;
    d.N = N;
    d.K = K;
    d.epi = EPI_STORE;
    gemm_tc_align(&d);
    int code = -1;
    std::vector<float> C(M * N);
    if (cudaMemcpy(dA, A.data(), A.size() * 2, cudaMemcpyHostToDevice) ||
        cudaMemcpy(dB, B.data(), B.size() * 2, cudaMemcpyHostToDevice) ||
        cudaMemcpy(dd, &d, sizeof d, cudaMemcpyHostToDevice))
      return 1;
    launch_gemm_tc(dd, dt, 1, 0, 0.f, err, 0);
    if (cudaMemcpy(C.data(), dC, M * N * 4, cudaMemcpyDeviceToHost) ||
        cudaMemcpy(&code, err, 4, cudaMemcpyDeviceToHost) || code)
      return 1;
    double tc = 0, chain = 0;
    for (int m = 0; m < M; ++m)
      for (int n = 0; n < N; ++n) {
        double s = 0;
        float f = 0;
        for (int k = 0; k < K; ++k) {
          const float a = __bfloat162float(A[m * K + k]), b = __bfloat162float(B[n * K + k]);
          s += (double)a * b;
          f = fmaf(a, b, f);
        }
        tc += (C[m * N + n] - s) * (C[m * N + n] - s);
        chain += (f - s) * (f - s);
      }
    printf("%d %.9g %.9g\n", K, std::sqrt(tc), std::sqrt(chain));
  }
  return 0;
}
"""


def test_products_are_as_exact_as_a_chain_of_fp32_additions(L, tmp_path_factory):  # noqa: F811
    """16384 products a length, so that each root mean square is known to half a percent."""
    out = run_program(native_program(tmp_path_factory, "gemm_error", PROGRAM,
                                     replaces=("gemm_tc.cu",)))
    rows = [tuple(map(float, r.split())) for r in out.splitlines()]
    assert len(rows) == 19
    for k, tc, chain in rows:
        assert tc <= 1.02 * chain, (k, tc, chain)

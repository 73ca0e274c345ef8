"""The meetings of the one-launch solves when a block never comes: the kernels compiled with a limit of 2000 polls run
with one block of the box left out, give up, set SC_KERR and end; the device stays usable."""
import ctypes
import subprocess

import pytest

from paper_1404_0959_gb300 import build as fe_build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#define FE_PK_SPINS 2000
#include "krylov_persist.cu"
namespace fe {
void prof_begin(Prof*, int, cudaStream_t) {}
void prof_end(Prof*, int, cudaStream_t) {}
__global__ void k_set(double* a, int n, double v, double w) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) a[i] = v + w * (i % 7);
}
}  // namespace fe
using namespace fe;

// scalars of the box after a solve at N = 16 with `missing` of its 32 blocks left out: iterations, converged, SC_KERR
extern "C" int run(int bicg, int missing, double* out) {
  const int N = 16, n = N * N * N, blocks = n / kPkThreads;
  const int slots[] = {K_B, W_DINV, W_PSI, K_AUX, K_PD, K_PP, K_X};
  BoxDev B;
  memset(&B, 0, sizeof(B));
  B.N = N;
  B.ih = N / (2.0 * M_PI);
  double *f = nullptr, *sums = nullptr, *coef = nullptr, sc[NSC] = {};
  unsigned* counters = nullptr;
  PkBlock* work = nullptr;
  BoxDev* box = nullptr;
  cudaMalloc(&f, sizeof(double) * (7 * n + NSC));
  cudaMalloc(&sums, sizeof(double) * 4 * blocks);
  cudaMalloc(&coef, sizeof(double) * kPkCoef * n);
  cudaMalloc(&counters, sizeof(unsigned) * kPkLine);
  cudaMalloc(&work, sizeof(PkBlock) * blocks);
  cudaMalloc(&box, sizeof(BoxDev));
  for (int q = 0; q < 7; ++q) B.f[slots[q]] = f + q * n;
  B.sc = f + 7 * n;
  sc[SC_KDT] = 0.1;
  sc[SC_TOL] = 1e-10;
  sc[SC_MAXIT] = 100;
  cudaMemcpy(B.sc, sc, sizeof(sc), cudaMemcpyHostToDevice);
  cudaMemcpy(box, &B, sizeof(B), cudaMemcpyHostToDevice);
  PkBlock w[64];
  for (int q = 0; q < blocks; ++q) w[q] = PkBlock{0, q, 1, 0, 0};
  cudaMemcpy(work, w, sizeof(PkBlock) * blocks, cudaMemcpyHostToDevice);
  cudaMemset(counters, 0, sizeof(unsigned) * kPkLine);
  cudaMemset(sums, 0, sizeof(double) * 4 * blocks);
  k_set<<<1, 256>>>((double*)B.f[K_B], n, -3.0, 1.0);
  k_set<<<1, 256>>>((double*)B.f[W_PSI], n, 1.0, 0.0);
  k_set<<<1, 256>>>((double*)B.f[W_DINV], n, 1.0 / (1.0 / 0.1 + 3.0 * 0.1 * B.ih * B.ih), 0.0);
  const BoxDev* boxes = box;
  void* args[] = {&boxes, &work, &sums, &counters, &coef};
  cudaLaunchCooperativeKernel((const void*)pk_kernel(bicg != 0, 1), dim3(blocks - missing), dim3(kPkThreads), args, 0, 0);
  const cudaError_t e = cudaDeviceSynchronize();
  cudaMemcpy(sc, B.sc, sizeof(sc), cudaMemcpyDeviceToHost);
  out[0] = sc[SC_ITERS];
  out[1] = sc[SC_CONV];
  out[2] = sc[SC_KERR];
  cudaFree(f), cudaFree(sums), cudaFree(coef), cudaFree(counters), cudaFree(work), cudaFree(box);
  return (int)e | (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    d = tmp_path_factory.mktemp("giveup")
    src, so = d / "giveup.cu", d / "giveup.so"
    src.write_text(SOURCE)
    subprocess.run([fe_build.nvcc()] + fe_build.ARCH + fe_build.FLAGS + ["-shared", "-I", fe_build.CSRC, str(src), "-o",
                                                                         str(so)], check=True)
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("bicg", [0, 1])
def test_a_block_that_never_comes(lib, bicg):
    out = (ctypes.c_double * 3)()
    for missing in (0, 1, 31, 0):
        assert lib.run(bicg, missing, out) == 0
        iters, conv, kerr = out
        if missing:
            assert kerr == 1.0 and conv == 0.0 and iters == 0.0
        else:
            assert kerr == 0.0 and conv == 1.0 and iters > 3

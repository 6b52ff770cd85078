"""Arithmetic of the tensor-core kernels one step at a time, through a small library that
calls the kernels' own functions on given operands.

Products (gemm_tc.cu), against exact integers.  In units of 2^{eA_i + eB_j}, where the
operands lie in (-1/4, 1/4): rounding both to multiples of 2^-64 adds at most
2 (1/4) 2^-65 + 2^-130 a term, the dropped digit pairs (7 of weight 2^-80, 6 of 2^-88, ...,
each at most 2^14) 7.03 2^-66, together 8.03 2^-66 for each of K terms; the result is
rounded once.  Row and column maxima are at least 1/8, so that this is below K 2^-56.99 of
(row max x column max).

Reflector norms (norm_and_gamma): the root is IEEE's, the reciprocal within 2 units of 2^-53."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include <cuda_bf16.h>
#include "common.cuh"
#include "tc_ptx.cuh"
using namespace dqmc;
__global__ void ng(const double* sig, const double* alpha, double* nrm, double* gam, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) norm_and_gamma(sig[i], alpha[i], nrm[i], gam[i]);
}
extern "C" int reflector(const double* sig, const double* alpha, double* nrm, double* gam, int n) {
  ng<<<(n + 255) / 256, 256>>>(sig, alpha, nrm, gam, n);
  return (int)cudaDeviceSynchronize();
}
extern "C" long long plane(int N, int R) { return tc_plane_elems(N, R); }
// C_b = A_b B_b of row-major N x N matrices; SA, SB, eA, eB as the splitter lays them out
extern "C" int product(const double* A, const double* B, double* out, int N, int batch, void* SA, void* SB,
                       int* eA, int* eB, int* status) {
  TcSplitArgs a;
  a.N = N; a.PM = (N + 31) / 32 * 32; a.sX = (long long)N * N;
  TcSplitArgs b = a;
  a.X = A; a.ldm = 1; a.ldj = N; a.R = 128; a.PJ = (N + 127) / 128 * 128;
  a.S = (__nv_bfloat16*)SA; a.sS = tc_plane_elems(N, 128); a.e = eA; a.se = a.PJ;
  b.X = B; b.ldm = N; b.ldj = 1; b.R = 64; b.PJ = (N + 63) / 64 * 64;
  b.S = (__nv_bfloat16*)SB; b.sS = tc_plane_elems(N, 64); b.e = eB; b.se = b.PJ;
  cudaError_t e;
  if ((e = tc_split(a, batch, nullptr)) != cudaSuccess || (e = tc_split(b, batch, nullptr)) != cudaSuccess) return (int)e;
  TcGemmArgs m;
  m.A = a.S; m.eA = eA; m.sA = a.sS; m.seA = a.se;
  m.B = b.S; m.eB = eB; m.sB = b.sS; m.seB = b.se;
  m.N = N; m.nkb = a.PM / 32; m.C = out; m.ldc = N; m.sC = (long long)N * N; m.status = status;
  if ((e = tc_gemm(m, batch, nullptr)) != cudaSuccess) return (int)e;
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def kit(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2003_05286_gb300 as m
    from paper_2003_05286_gb300 import build as b
    m.lib()
    lib, d = b.lib_path(), tmp_path_factory.mktemp("kit")
    (d / "kit.cu").write_text(SRC)
    subprocess.run([b._nvcc(), *b.ARCH, *b.FLAGS, "-shared", "-I", os.path.join(ROOT, "include"), "-I", b.CSRC,
                    str(d / "kit.cu"), lib, "-Xlinker", "-rpath," + os.path.dirname(lib), "-o", str(d / "kit.so")],
                   check=True)
    kit = C.CDLL(str(d / "kit.so"))
    kit.plane.restype = C.c_longlong
    return kit


def _p(t):
    return C.c_void_p(t.data_ptr())


def _exact(x):
    """Integers and a common power of two: x = n 2^-s (entries below FP64's largest digits
    by at most 1100 bits)."""
    m, e = np.frexp(x)
    s = int(53 - e[x != 0].min()) if (x != 0).any() else 0
    return [int(v * 2.0 ** 53) << (int(k) - 53 + s) if v else 0 for v, k in zip(m.ravel(), e.ravel())], s


def _operands(kind, N, rng):
    A, B = rng.standard_normal((2, 2, N, N))
    if kind == "digits":            # one entry of order one a row, the others with all low digits -128
        low = -4 * sum(2.0 ** (-8 * p - 1) for p in range(1, 8))       # (scaled by 2^-2)
        A, B = np.full((2, N, N), low), np.full((2, N, N), -low)
        A[:, :, 0], B[:, 0, :] = 0.9375, 0.96875
    if kind == "graded":            # rows of A and columns of B over many orders, entries too
        A = A * np.exp(rng.uniform(-200, 200, (2, N, 1)) + rng.uniform(-30, 0, (2, N, N)))
        B = B * np.exp(rng.uniform(-200, 200, (2, 1, N)) + rng.uniform(-30, 0, (2, N, N)))
    if kind == "tiny":              # products in the subnormal range
        A, B = A * 2.0 ** -700, B * 2.0 ** -345
    return A, B


@pytest.mark.parametrize("kind", ["normal", "digits", "graded", "tiny"])
@pytest.mark.parametrize("N", [64, 129, 256, 257, 768])
def test_product(kit, N, kind):
    rng = np.random.default_rng(N)
    A, B = _operands(kind, N, rng)
    dev = lambda x: torch.tensor(np.ascontiguousarray(x), device="cuda")
    Ad, Bd, out = dev(A), dev(B), torch.empty(2, N, N, dtype=torch.float64, device="cuda")
    SA = torch.empty(2 * kit.plane(N, 128), dtype=torch.bfloat16, device="cuda")
    SB = torch.empty(2 * kit.plane(N, 64), dtype=torch.bfloat16, device="cuda")
    eA, eB, st = (torch.zeros(n, dtype=torch.int32, device="cuda") for n in (2 * (N + 127), 2 * (N + 63), 2))
    assert kit.product(_p(Ad), _p(Bd), _p(out), N, 2, _p(SA), _p(SB), _p(eA), _p(eB), _p(st)) == 0
    assert int(st.sum()) == 0
    got = out.cpu().numpy()
    for _ in range(60):
        b, i, j = rng.integers(0, 2), rng.integers(0, N), rng.integers(0, N)
        (x, sx), (y, sy) = _exact(A[b, i]), _exact(B[b, :, j])
        z, s = sum(p * q for p, q in zip(x, y)), sx + sy
        # exponents of the row and the column: the largest entry in [1/8, 1/4)
        ea = int(np.frexp(A[b, i])[1].max()) + 2
        eb = int(np.frexp(B[b, :, j])[1].max()) + 2
        g, sg = _exact(got[b, i, j:j + 1])
        top = max(s, sg, 70 - ea - eb, 1140)
        err = abs((g[0] << (top - sg)) - (z << (top - s)))
        bound = (N * 803 << (top + ea + eb - 66)) // 100 if top + ea + eb >= 66 else 0
        half = 1 << (top - 1075)                     # half the last place of the result, at least 2^-1075
        v = abs(got[b, i, j])
        if v >= 2.0 ** -1022:
            half = 1 << (top + int(np.frexp(v)[1]) - 54)
        assert err <= bound + half + 1, (b, i, j)


def test_reflector_norm_and_reciprocal(kit):
    rng = np.random.default_rng(3)
    n = 1 << 20
    sig = rng.uniform(1, 4, n) * 2.0 ** rng.integers(-960, 994, n)
    alpha = np.sqrt(sig) * np.where(rng.random(n) < 0.1, 1.0, rng.uniform(0, 1, n)) * rng.choice([-1.0, 1.0], n)
    sig[:3], alpha[:3] = [1.0, 4.0, 2.0], [1.0, 0.0, -np.sqrt(2.0)]
    d = [torch.tensor(x, device="cuda") for x in (sig, alpha)] + [torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2)]
    assert kit.reflector(*map(_p, d), n) == 0
    nrm, gam = d[2].cpu().numpy(), d[3].cpu().numpy()
    assert (nrm == np.sqrt(sig)).all()
    # (longdouble has at least 64 bits on both of the machines in use)
    want = 1 / (sig.astype(np.longdouble) + np.abs(alpha).astype(np.longdouble) * nrm)
    assert float(np.abs(gam / want - 1).max()) <= 2.0 * 2.0 ** -53

"""The training forward's sums against exact rational arithmetic on the same FP32
factors: as many bits as FP64 sums of the terms would have, at any eps_k and scale, and
finite where only the products (not the score) leave the range of FP32.

Tolerance: a term is carried to 2^-53 of itself, and three FP64 roundings follow, each
2^-53 of at most the sum of the terms' magnitudes: below 2^-51 of that sum.  At the
scale where the products leave the range of FP32 the terms are summed in FP64: one
rounding of 2^-53 for each term and three for its factors."""

import math
import struct
import subprocess
from fractions import Fraction

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

POINTS, TERMS = 96, 31

PROGRAM = r"""
#include "gd_leaf_kernel.cuh"
#include <cstdio>
#include <cstdlib>
using namespace gd;
constexpr uint32_t N = %d, T = %d;
__global__ void k_sums(LeafArgs A, const float *in, float *factors, int any) {  // one point a thread
  const uint32_t i = threadIdx.x;
  if (i >= N) return;
  const float *x = in + (size_t)i * (2 + 2 * T);  // ell_i, c_i, then (d^2, ell_j)
  TrainSums s;
  TrainSumsAny sx;
  float F = 0.0f;
  for (uint32_t j = 0; j < T; ++j) {
    const float d2 = x[2 + 2 * j], lj = x[3 + 2 * j], q = __fadd_rn(d2, A.p.eps_k);
    s.add(A.p, true, d2, x[0], lj, x[1]);
    sx.add(A.p, true, d2, x[0], lj, x[1]);
    float *f = factors + ((size_t)i * T + j) * 3;  // the term's factors, as the sums take them
    f[0] = __fdiv_rn(exp2f(__fmaf_rn(__fmul_rn(0.5f, A.p.alpha), __fadd_rn(x[0], lj), -__fmul_rn(d2, x[1]))), q);
    f[1] = __fmul_rn(__fadd_rn(x[0], lj), 0.6931471805599453f);
    f[2] = d2 > 0.0f ? logf(d2) : 0.0f;
  }
  for (uint32_t j = 0; j < T; ++j) F += factors[((size_t)i * T + j) * 3];
  if (any || !s.fits(A.p, F)) sx.store(A, i, 1.0f);
  else s.store(A, i, 1.0f);
}
int main(int, char **v) {
  LeafArgs A{};
  A.n = N;
  A.p.alpha = 1.3f;
  A.p.gamma = 2.0f;
  A.p.eps_k = (float)atof(v[1]);
  float *in, *f;
  const size_t nin = (size_t)N * (2 + 2 * T), nf = (size_t)N * T * 3;
  cudaMallocManaged(&in, 4 * nin);
  cudaMallocManaged(&f, 4 * nf);
  cudaMallocManaged(&A.train.sums, 24 * N);
  cudaMallocManaged(&A.train.r2, 4 * N);
  cudaMallocManaged(&A.ctr, sizeof(Counters));
  FILE *h = fopen(v[2], "rb");
  if (!h || fread(in, 4, nin, h) != nin) return 2;
  fclose(h);
  k_sums<<<1, 128>>>(A, in, f, atoi(v[4]));
  if (cudaDeviceSynchronize() != cudaSuccess) return 3;
  h = fopen(v[3], "wb");
  fwrite(A.train.sums, 24, N, h);
  fwrite(f, 4, nf, h);
  fclose(h);
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    from paper_2512_10386_gb300 import build
    d = tmp_path_factory.mktemp("sums")
    (d / "sums.cu").write_text(PROGRAM % (POINTS, TERMS))
    subprocess.run([build._nvcc(), *build.NVCC_FLAGS, str(d / "sums.cu"), "-o", str(d / "sums")], check=True)
    return d


@pytest.mark.parametrize("any_term", [0, 1])
@pytest.mark.parametrize("scale", [1e-35, 1e-12, 1e-4, 1.0, 1e10])
@pytest.mark.parametrize("eps", [0.0, 1e-12, 1e-9, 1e-4, 1.0])
def test_bits(program, scale, eps, any_term):
    g = torch.Generator().manual_seed(int(1e3 * eps) + POINTS)
    x = torch.empty(POINTS, 2 + 2 * TERMS)
    x[:, 0] = torch.randn(POINTS, generator=g)
    d2 = scale * torch.rand(POINTS, TERMS, generator=g) ** 2 + 1e-2 * scale
    if eps > 0:
        d2[:, 3] = 0.0  # a duplicate of the point
    x[:, 1] = 0.72 / d2.amax(1)
    x[:, 2::2] = d2
    x[:, 3::2] = torch.randn(POINTS, TERMS, generator=g)
    (program / "in").write_bytes(x.numpy().tobytes())
    subprocess.run([str(program / "sums"), repr(eps), str(program / "in"), str(program / "out"),
                    str(any_term)], check=True)
    raw = (program / "out").read_bytes()
    sums = struct.unpack(f"<{3 * POINTS}d", raw[:24 * POINTS])
    fac = struct.unpack(f"<{3 * POINTS * TERMS}f", raw[24 * POINTS:])
    ek = Fraction(float(torch.tensor(eps)))
    bits = Fraction(TERMS + 6, 2 ** 53) if scale == 1e-35 else Fraction(1, 2 ** 51)
    for i in range(POINTS):
        terms = []
        for j in range(TERMS):
            t, lw, l = (Fraction(v) for v in fac[3 * (i * TERMS + j):3 * (i * TERMS + j) + 3])
            d = Fraction(float(x[i, 2 + 2 * j]))
            terms.append((t * lw, t * d, t * l * (d / (d + ek) if d else 0)))
        for q in range(3):
            exact, mag = sum(v[q] for v in terms), sum(abs(v[q]) for v in terms)
            assert abs(Fraction(sums[3 * i + q]) - exact) <= mag * bits, (i, q)


def test_products_beyond_fp32_stay_finite():
    """eps_k = 0 and squared distances near 1e-36: the score fits FP32, the terms' products
    with ln W and ln d^2 do not.  A cloud scaled by a power of two has the same gates and
    neighbours; alpha and sigma see ratios of distances only, every ln d^2 of gamma's sum
    is shifted by 2 ln(scale)."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_10386_gb300 import Denoiser, Params
    a = torch.arange(16, dtype=torch.float32)
    xyz = torch.stack(torch.meshgrid(a, a, a, indexing="ij"), -1).reshape(-1, 3)
    xyz = (xyz + 0.4 * torch.rand(xyz.shape, generator=torch.Generator().manual_seed(2))).cuda()
    n, scale, got = len(xyz), 2.0 ** -60, []
    for s in (1.0, scale):
        d = Denoiser(max_points=n)
        try:
            d.set_training(True)
            d.run(xyz * s, Params(k=12, select_mode=1, eps_k=0.0, eps_rho=0.0, min_vox_count=1,
                                  tau=2.0 - 2.0 * math.log(s), temperature=1.0))
            got.append(d.backward(torch.ones(n, device="cuda")))
        finally:
            d.close()
    a, b = got
    for q in (0, 1, 3):  # (FP32 factors, ln F - tau at |tau| = 81: 1e-5 each)
        assert b[q] == pytest.approx(a[q], rel=1e-3)
    assert b[2] == pytest.approx(a[2] + math.log(scale) * a[3], rel=1e-3)

"""The tensor-core exact attention at the edges of its layout: every window
size it takes, the narrowest and widest heads (padding columns, the ones column
inside and beyond them), one unit up to several rounds of groups, fp32's split
planes, and rows whose scores differ by far more than the exponential's range."""
import numpy as np
import pytest
import torch

import oracle
from paper_2506_08520_gb300 import binding, workloads
from tests.parity import ROUND, TOL, per_unit_rel, units_view

pytestmark = pytest.mark.gpu

# P and the output are rounded to 16 bits; fp32 I/O takes 16-bit pairs
BAR = {"f32": TOL["f32"], "bf16": 2 * ROUND["bf16"], "f16": 2 * ROUND["f16"]}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2506_08520_gb300 import build
    build.build()


def _check(q, k, v, tol):
    out = binding.exact(q.cuda(), k.cuda(), v.cuda())
    torch.cuda.synchronize()
    err = per_unit_rel(units_view(out.cpu()).double().numpy(), oracle.exact_attention(q, k, v))
    assert err.max() <= tol, f"{err.max():.3e} at unit {int(np.argmax(err))}"


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("units,N,d", [(1, 64, 2), (1825, 64, 30), (3, 64, 32), (2, 64, 24), (1, 256, 2),
                                       (609, 256, 30), (2, 256, 32), (3, 256, 18), (1, 1024, 30), (2, 1024, 32),
                                       (3, 1024, 8)])
def test_units_and_widths(units, N, d, dtype):
    if N == 1024 and dtype == "f32":
        pytest.skip("32x32 windows in fp32 take the generic kernel")
    q, k, v = workloads.random_qkv(units, N, d, dtype, seed=units + N + d)
    _check(q, k, v, BAR[dtype])


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("d", range(2, 33, 2))
def test_every_head_width(d, dtype):
    # rows of d / 2 words laid out in batches, d read at run time but for 30 and 32;
    # one group per CTA, and (457 units) up to four, the last one idle in some
    for units, N in ((5, 64), (457, 64), (2, 256)):
        q, k, v = workloads.random_qkv(units, N, d, dtype, seed=units + N + d)
        _check(q, k, v, BAR[dtype])


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("N", [64, 256])
def test_late_maximum(N, dtype):
    # the row maximum sits in the last key chunk and exceeds every earlier
    # score by about 50: the accumulated rows are rescaled to nothing
    q, k, v = workloads.random_qkv(2, N, 30, "f32", seed=N)
    T = workloads.DTYPES[dtype]
    k[:, -1] = 0.0
    q[..., 0], k[..., 0] = 4.0, torch.linspace(-30, 30, N)
    _check(q.to(T), k.to(T), v.to(T), BAR[dtype])


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("units,N,d", [(2, 1, 1), (3, 63, 16), (3, 64, 17), (2, 65, 20), (2, 127, 21), (2, 129, 33),
                                       (3, 200, 36), (2, 256, 37), (2, 100, 64), (1, 1024, 30), (1, 1000, 63),
                                       (5, 4, 16), (2, 15, 33), (3, 16, 20), (2, 16, 64), (2, 17, 30)])
def test_generic_tile_edges(units, N, d, dtype):
    # blocks of 64 rows and chunks of 64 keys, one more or less than whole
    # ones, and the single ones of 16 that small windows take; the head widths at which row strides and key splits change
    q, k, v = workloads.random_qkv(units, N, d, dtype, seed=units + N + d)
    # fp32 throughout: a few ulp of the longest sums (2^-24 x sqrt(1024) = 2e-6)
    _check(q, k, v, 2e-6 if dtype == "f32" else ROUND[dtype])


def _rounded_p(q, k, v, chunk):
    """Eq. 1 with the online softmax over chunks of keys: float64 but for P,
    rounded to the I/O type relative to the running maximum, and the result."""
    T = q.dtype
    q, k, v = q.double(), k.double(), v.double()
    N, d = q.shape[1:]
    s = torch.einsum("utd,ukd->utk", q, k) * (1.4426950408889634 / d ** 0.5)
    run = torch.full(s.shape[:2] + (1,), -float("inf"), dtype=torch.float64)
    num, den = torch.zeros_like(q), torch.zeros_like(run)
    for c in range(0, N, chunk):
        m = torch.maximum(run, s[..., c:c + chunk].amax(-1, keepdim=True))
        f, p = torch.exp2(run - m), torch.exp2(s[..., c:c + chunk] - m).to(T).double()
        num, den, run = num * f + p @ v[:, c:c + chunk], den * f + p.sum(-1, keepdim=True), m
    return (num / den).to(T).double()


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("units,N,d", [(6, 256, 30), (6, 256, 32), (6, 256, 18), (2, 1024, 30), (2, 1024, 32), (2, 1024, 8)])
def test_probabilities_are_rounded_at_the_maxima_of_64_keys(units, N, d, dtype):
    # another chunk length rounds other values: the results lie some 2^-9 apart in
    # bf16, 2^-12 in fp16, and fp32 sums and ex2 move at most a quarter of that
    # (fp16, 1024 keys: a relative 2^-22 of P moves one value in 500 to its
    # neighbour).  Within half of it, the output belongs to the one and not the other
    q, k, v = workloads.random_qkv(units, N, d, dtype, seed=N + d)
    out = units_view(binding.exact(q.cuda(), k.cuda(), v.cuda()).cpu()).double()
    ref, other = _rounded_p(q, k, v, 64), _rounded_p(q, k, v, 32)
    assert (out - ref).norm() <= 0.5 * (other - ref).norm()

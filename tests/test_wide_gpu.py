"""The wide-landmark kernel (m = 64 at 8x8 and 16x16 windows) and its core of
symmetric products: one group up to many, no steps to many, the narrowest and
widest heads, and columns of V of very different scales."""
import numpy as np
import pytest
import torch

import oracle
from paper_2506_08520_gb300 import binding, workloads
from tests.parity import ROUND, TOL, per_unit_rel, units_view

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2506_08520_gb300 import build
    build.build()


def _run(q, k, v, iters, factors="pairs"):
    out = binding.nystra(q.cuda(), k.cuda(), v.cuda(), 64, iters, factors=factors)
    torch.cuda.synchronize()
    assert binding.status() == binding.NYSTRA_OK
    return units_view(out.cpu()).double().numpy()


@pytest.mark.parametrize("factors", ["pairs", "16"])
@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("units,N,d,iters", [(1, 64, 30, 6), (461, 64, 2, 5), (7, 64, 32, 0), (2, 256, 30, 0),
                                             (3, 256, 32, 1), (460, 256, 16, 2), (5, 256, 2, 6), (2, 1024, 30, 1),
                                             (3, 1024, 32, 0)])
def test_units_steps_and_widths(units, N, d, iters, dtype, factors):
    q, k, v = workloads.random_qkv(units, N, d, dtype, seed=N + d + iters)
    err = per_unit_rel(_run(q, k, v, iters, factors), oracle.nystra_attention(q, k, v, 64, iters))
    # single 16-bit factors: G_L, G_U, the landmarks and Y are rounded too
    assert err.max() <= (1 if factors == "pairs" else 5) * ROUND[dtype], f"{err.max():.3e} at unit {int(np.argmax(err))}"


@pytest.mark.parametrize("dtype,lo,hi", [("bf16", -30, 30), ("f16", -10, 5)])
@pytest.mark.parametrize("N", [64, 256, 1024])
def test_columns_of_any_scale(N, dtype, lo, hi):
    # V's columns are independent outputs: scaling one by a power of two (exact
    # in the I/O type) scales that output column and leaves the others alone,
    # whatever the range between the columns and the ones column
    q, k, v = workloads.random_qkv(4, N, 30, "f32", seed=N)
    T = workloads.DTYPES[dtype]
    q, k = q.to(T), k.to(T)
    v = (v.clamp(-3, 3).sign() * (v.abs().clamp(0.25, 3))).to(T)
    s = torch.pow(2.0, torch.linspace(lo, hi, 30).round())
    a = _run(q, k, v, 6)
    b = _run(q, k, (v.float() * s).to(T), 6) / s.double().numpy()
    ref = oracle.nystra_attention(q, k, v, 64, 6)
    col = np.linalg.norm(b - ref, axis=1) / np.linalg.norm(ref, axis=1)
    # fp16 outputs below 2^-14 are subnormal: 2^-25 absolute on outputs of about 0.1 2^lo;
    # and Y^T's fp16 pairs, at one scale, end 2^-39 below its largest entry, 2^-24 below
    # those of the smallest column, which Z may exceed the output 10^4 times
    bar = ROUND[dtype] if dtype == "bf16" else TOL[dtype] + 2.0 ** -25 / (0.02 * 2.0 ** lo)
    assert col.max() <= bar, col.max()
    assert per_unit_rel(a, ref).max() <= ROUND[dtype]


@pytest.mark.parametrize("N,m", [(64, 32), (64, 64), (256, 32), (256, 64), (1024, 32), (1024, 64)])
def test_landmarks_of_any_scale(N, m):
    # two groups of tokens that attend to their own group alone: feature 0 is +20 or
    # -20, so a score across is 146 below one within and its exponential 0 in fp32.
    # The rows of V (and of W) of one group are scaled by 2^-40, exact in bf16: so
    # is its output, to all its digits, whatever the other group's rows of W hold
    q, k, v = (x.bfloat16() for x in workloads.random_qkv(3, N, 30, "f32", seed=N + m))
    near = torch.arange(N) < N // 2
    for x in (q, k):
        x[..., 0] = torch.where(near, 20.0, -20.0)
    s = torch.where(near, 2.0 ** -40, 1.0)[:, None]
    out = binding.nystra(q.cuda(), k.cuda(), (v.float() * s).bfloat16().cuda(), m, 6)
    torch.cuda.synchronize()
    assert binding.status() == binding.NYSTRA_OK
    out = units_view(out.cpu()).double().numpy() / s.double().numpy()
    ref = oracle.nystra_attention(q, k, v, m, 6)
    for rows in (slice(0, N // 2), slice(N // 2, N)):
        assert per_unit_rel(out[:, rows], ref[:, rows]).max() <= ROUND["bf16"]

"""The generic kernel at the edges of its tiles: token chunks of 160, 128 and
64 rows (one more or less than whole ones), groups of four tokens, landmarks
and columns, the three row strides (d_h up to 19, 35 and 64) and the landmark
bounds 8, 16, 32 and 64, against the float64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2506_08520_gb300 import binding, workloads
from tests.parity import ROUND, TOL, nystra_float32, per_unit_rel, units_view

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2506_08520_gb300 import build
    build.build()


SHAPES = [  # N, d, m, pooling
    (5, 3, 5, "segments"), (9, 4, 1, "patches"), (49, 32, 7, "segments"), (160, 19, 8, "segments"),
    (161, 20, 7, "segments"), (320, 36, 8, "segments"), (81, 16, 9, "patches"), (159, 31, 3, "segments"),
    (162, 35, 9, "segments"), (324, 64, 12, "segments"), (1024, 17, 16, "patches"), (130, 36, 26, "segments"),
    (128, 63, 32, "segments"), (1020, 30, 17, "segments"), (64, 30, 64, "patches"), (66, 64, 33, "segments"),
    (1024, 64, 64, "segments"), (63, 2, 63, "segments"), (576, 32, 36, "patches"),
]


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("N,d,m,pool", SHAPES)
def test_generic_tile_edges(N, d, m, pool, dtype):
    q, k, v = workloads.random_qkv(3, N, d, dtype, seed=N + 7 * d + m)
    out = binding.nystra(q.cuda(), k.cuda(), v.cuda(), m, 5, landmarks=pool)
    torch.cuda.synchronize()
    err = per_unit_rel(units_view(out.cpu()).double().numpy(), oracle.nystra_attention(q, k, v, m, 5, pool))
    bar = np.full(3, ROUND[dtype])
    if dtype == "f32" and pool == "segments":
        # fp32 throughout: within the float32 evaluation's own error (4x: another
        # order of sums) or 2^-24 per step of the longest sum, at least 1e-6
        ref = oracle.nystra_attention(q, k, v, m, 5)
        bar = np.minimum(bar, np.maximum(4.0 * per_unit_rel(nystra_float32(q, k, v, m, 5), ref), 1e-6))
    assert (err <= bar).all(), f"{err} > {bar}"


@pytest.mark.parametrize("N,d,m,per_window", [(162, 33, 9, False), (100, 20, 20, True), (64, 64, 64, False)])
def test_generic_score_bias(N, d, m, per_window):
    rng = np.random.default_rng(N + m)
    q, k, v = (x.reshape(3, 2, N, d) for x in workloads.random_qkv(6, N, d, "f32", seed=N + d))
    B = torch.from_numpy(0.5 * rng.standard_normal(((3, 2) if per_window else (2,)) + (N, N))).float()
    pooled = binding.pool_bias(B.cuda(), m)
    out = binding.nystra_biased(q.cuda(), k.cuda(), v.cuda(), pooled, m, 5)
    torch.cuda.synchronize()
    ref = oracle.nystra_attention(q, k, v, m, 5, "segments", B.double().numpy() if per_window else B.double().numpy()[None])
    err = per_unit_rel(out.cpu().double().numpy(), ref)
    assert err.max() <= TOL["f32"], err


@pytest.mark.parametrize("N,d,m", [(5, 3, 5), (49, 30, 7), (36, 20, 4), (81, 16, 9)])
def test_generic_few_and_many_units(N, d, m):
    # up to four units per SM (608 on 152 SMs) a CTA has four warps at least, above
    # only its tiles' threads: the sums are the same
    q, k, v = workloads.random_qkv(609, N, d, "f32", seed=N + d)
    out = binding.nystra(q.cuda(), k.cuda(), v.cuda(), m, 5)
    few = binding.nystra(q[1:].cuda(), k[1:].cuda(), v[1:].cuda(), m, 5)
    torch.cuda.synchronize()
    assert torch.equal(out[1:], few)
    at = [0, 304, 608]
    q, k, v = q[at], k[at], v[at]
    ref = oracle.nystra_attention(q, k, v, m, 5)
    err = per_unit_rel(units_view(out[at].cpu()).double().numpy(), ref)
    bar = np.maximum(4.0 * per_unit_rel(nystra_float32(q, k, v, m, 5), ref), 1e-6)  # as above
    assert (err <= np.minimum(bar, TOL["f32"])).all(), f"{err} > {bar}"

"""Heads of 32 features in 16 bits, whose rows the kernels read and write 16
bytes at a time: every feature's place, on one unit up to a ragged number."""
import numpy as np
import pytest
import torch

import oracle
from paper_2506_08520_gb300 import binding, workloads
from tests.parity import ROUND, per_unit_rel, units_view

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2506_08520_gb300 import build
    build.build()


@pytest.mark.parametrize("factors", ["pairs", "16"])
@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("units,N,m", [(1, 64, 8), (149, 64, 16), (3, 64, 64), (2, 256, 8), (155, 256, 16), (5, 256, 32),
                                       (2, 256, 64), (1, 1024, 8), (153, 1024, 16), (3, 1024, 32), (2, 64, 32)])
def test_every_feature_keeps_its_place(units, N, m, dtype, factors):
    # features of unequal weight in the scores (Q times sqrt(weight), K too) and
    # columns of V apart by exact powers of two: a feature in another's place shows
    q, k, v = workloads.random_qkv(units, N, 32, "f32", seed=N + m)
    T = workloads.DTYPES[dtype]
    w = torch.linspace(0.25, 1.5, 32)
    q, k = (q * w).to(T), (k * w).to(T)
    s = torch.pow(2.0, (torch.arange(32) % 7 - 3).float())
    v = (v.to(T).float() * s).to(T)
    out = binding.nystra(q.cuda(), k.cuda(), v.cuda(), m, 6, factors=factors)
    torch.cuda.synchronize()
    assert binding.status() == binding.NYSTRA_OK
    out = units_view(out.cpu()).double().numpy() / s.double().numpy()
    ref = oracle.nystra_attention(q, k, v, m, 6) / s.double().numpy()
    err = per_unit_rel(out, ref)
    # single 16-bit factors: G_L, G_U, the landmarks and Y are rounded too
    bar = (1 if factors == "pairs" else 5) * ROUND[dtype]
    assert err.max() <= bar, f"{err.max():.3e} at unit {int(np.argmax(err))}"
    col = np.linalg.norm(out - ref, axis=(0, 1)) / np.linalg.norm(ref, axis=(0, 1))
    # a column's own error: rounding of the output and of W's column, as for the whole
    assert col.max() <= 2 * bar, col.max()

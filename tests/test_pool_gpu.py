"""The 8x8-window kernel, whose warps keep landmarks, W, Y^T and output rows
one after the other in the same memory: a unit's result is the same bits
wherever it lies in a call, up to more units than warps on the GPU."""
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


@pytest.mark.parametrize("biased", [False, True])
@pytest.mark.parametrize("d,m,dtype,pool", [(30, 16, "bf16", "segments"), (30, 16, "f16", "patches"), (30, 8, "bf16", "segments"),
                                            (32, 16, "f16", "segments"), (32, 8, "bf16", "segments"),
                                            (32, 16, "bf16", "patches"), (24, 16, "bf16", "segments"),
                                            (2, 8, "f16", "segments"), (30, 16, "f32", "segments"),
                                            (32, 8, "f32", "segments"), (18, 16, "f32", "segments")])
def test_a_unit_is_the_same_anywhere(d, m, dtype, pool, biased):
    n = 7
    q, k, v = workloads.random_qkv(n, 64, d, dtype, seed=d + m)
    B = torch.from_numpy(0.5 * np.random.default_rng(m).standard_normal((1, 64, 64))).float()
    pooled = binding.pool_bias(B.cuda(), m, landmarks=pool) if biased else None

    def run(u):
        a, b, c = (x.cuda()[torch.arange(u, device="cuda") % n].view(u, 1, 64, d) for x in (q, k, v))
        out = (binding.nystra_biased(a, b, c, pooled, m, 6, landmarks=pool) if biased else
               binding.nystra(a, b, c, m, 6, landmarks=pool))
        torch.cuda.synchronize()
        assert binding.status() == binding.NYSTRA_OK
        return out.view(u, 64, d)

    few = run(n)
    ref = oracle.nystra_attention(q, k, v, m, 6, pool, B.double().numpy()) if biased else \
        oracle.nystra_attention(q, k, v, m, 6, pool)
    err = per_unit_rel(units_view(few.cpu()).double().numpy(), np.asarray(ref).reshape(n, 64, d))
    assert err.max() <= ROUND[dtype], err
    for u in (1, 16, 2 * 152 * 16 + 5):
        many = run(u)
        assert torch.equal(many, few[torch.arange(u, device="cuda") % n])

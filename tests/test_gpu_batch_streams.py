"""Batched solves whose plans share the caller's stream: they run side by
side, and a solve that starts from another one's result still follows it."""
import numpy as np
import pytest

from paper_0908_3252_gb300 import synth
from tests.helpers import empty_c64, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chained", [False, True])
def test_batch_on_one_stream(chained):
    import torch
    from paper_0908_3252_gb300 import build, spirec as sp
    build.build()
    plans, singles = [], []
    g = synth.rng(5)
    kx, ky = synth.uniform_k(900, g)
    for _ in range(3):
        p = sp.Plan(32, 900, 0, sp.SPIREC_MIXED_FP16X3, torch.cuda.current_stream().cuda_stream, kx, ky)
        sp.spirec_set_data(p.h, synth.complex_normal(900, g).astype(np.complex64))
        sp.spirec_set_reg(p.h, 0.05, 0.05, 0.02, 0.1, 0)
        plans.append(p)
    start = to_dev(synth.complex_normal((32, 32), g))
    prev = start
    for p in plans:
        x = empty_c64((32, 32))
        sp.spirec_solve_dev(p.h, prev, 4, x, None)
        torch.cuda.synchronize()
        singles.append(x)
        prev = x if chained else start
    outs = [empty_c64((32, 32)) for _ in plans]
    sp.spirec_batch_solve([p.h for p in plans], outs, 4, x0=[start] + (outs[:-1] if chained else [start] * 2))
    torch.cuda.synchronize()
    for x, y in zip(singles, outs):
        assert torch.equal(x, y)
    for p in plans:
        p.close()

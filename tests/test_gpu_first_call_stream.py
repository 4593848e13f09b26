"""A context's first calls on a stream of their own while the default stream is busy:
what its new buffers have to start with is ordered before the calls that read it, not
behind the default stream's work. (New device memory may happen to hold zeros: the
order itself is checked on the source, tests/test_stream_order.py.)"""
import numpy as np
import pytest
import torch

import oracle
from tests import _systems as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1607_02904_gb300 as T
    T.load()
    return T


def used_memory():
    a = [torch.full((1 << 18,), 7.25, dtype=torch.float64, device="cuda") for _ in range(40)]
    torch.cuda.synchronize()
    del a
    torch.cuda.empty_cache()


@pytest.mark.parametrize("scatter", [0, 1], ids=["gather", "atomic"])
@pytest.mark.parametrize("switch", [False, True], ids=["one-precision", "precision-switched"])
def test_new_buffers(T, scatter, switch):
    x, t, box = S.sic_cell(n=8, sigma=0.1, seed=701)
    table = S.table_for(["Si", "C"], oracle.mix_tersoff89)
    ref = oracle.compute(x, t, box, table, oracle.neighbors(x, box, 3.0))[1]
    xd, td = torch.tensor(x, device="cuda"), torch.tensor(t, dtype=torch.int32, device="cuda")
    f = [torch.zeros_like(xd) for _ in range(3)]
    side = torch.cuda.Stream()
    ctx = T.Context(T.FP64)
    ctx.set_scatter(scatter)
    ctx.params(table)
    used_memory()
    torch.cuda._sleep(400_000_000)  # the default stream, some 200 ms
    with torch.cuda.stream(side):
        ctx.neighbor_build(xd, td, box, 4.0)
        ctx.compute(xd, None, f[0])
        if switch:
            ctx.set_precision(T.MIXED)
            ctx.compute(xd, None, f[1])
            ctx.set_precision(T.FP64)
        ctx.compute(xd, None, f[2])
    side.synchronize()
    torch.cuda.synchronize()
    for k, tol in ((0, 1e-10), (2, 1e-10)) + (((1, 1e-4),) if switch else ()):
        assert np.abs(f[k].cpu().numpy() - ref).max() <= tol * np.abs(ref).max()
    ctx.close()

"""The wide launch beside the main one (bucket 2 on a stream of its own), with and
without the capacity-8 launch split off: repeated calls, calls on another stream,
and a captured graph's replay give the same forces bit for bit, and match the
oracle (mixed path, relative force RMS 1e-5)."""
import numpy as np
import pytest
import torch

import oracle
from tests import _systems as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [-1, 0, 1])
def test_streams_and_capture(split):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1607_02904_gb300 as T
    T.load()
    x, t, box = S.sic_cell(n=8, sigma=0.12, seed=701)
    table = S.table_for(["Si", "C"], oracle.mix_tersoff89)
    c = T.Context(T.MIXED)
    c.set_launch(split=split)
    c.params(table)
    xd = torch.tensor(x, device="cuda")
    c.neighbor_build(xd, torch.tensor(t, dtype=torch.int32, device="cuda"), box, 4.0)
    f = torch.zeros_like(xd)
    e = torch.zeros(1, dtype=torch.float64, device="cuda")
    c.compute(xd, e, f)
    torch.cuda.synchronize()
    first = f.clone()
    ref = oracle.compute(x, t, box, table, oracle.neighbors(x, box, 3.1))
    fr = first.cpu().numpy()
    assert np.sqrt(((fr - ref[1]) ** 2).sum() / (ref[1] ** 2).sum()) <= 1e-5
    side = torch.cuda.Stream()
    for _ in range(3):
        with torch.cuda.stream(side):
            f.zero_()
            c.compute(xd, e, f, stream=side)
        side.synchronize()
        assert torch.equal(f, first)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        c.compute(xd, e, f, stream=torch.cuda.current_stream())
    for _ in range(3):
        f.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(f, first)
    c.close()

"""The FP64 path's parameter adjoint of one species at the largest size that takes
eight lanes per atom and the next: against the oracle's complex step (1e-10 of
the largest entry, each scaled by its parameter), with and without lambda3."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from tests import _systems as S
from tests.test_gpu_backward import scaled_err, weights

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lam3", [False, True])
@pytest.mark.parametrize("cells", [(5, 10, 25), (3, 3, 139)], ids=["10000", "10008"])
def test_one_species_by_size(cells, lam3):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1607_02904_gb300 as T
    T.load()
    x, t, box = W.diamond(*cells, 5.432)
    x = W.jitter_gaussian(x, 0.08, np.random.Generator(np.random.Philox(801)))
    table = S.table_for(["Si"], oracle.mix_tersoff89)
    if lam3:
        table = S.with_lambda3(table, 1.7322, 3)
    gE, gF = weights(len(x), 802)
    nl = oracle.neighbors(x, box, 3.0)
    ref = np.zeros(table.size)
    for p in range(1, table.size):
        de, df = oracle.cs_param(x, t, box, table, nl, p)
        ref[p] = gE * de + float((gF * df).sum())
    c = T.Context(T.FP64)
    c.params(table)
    xd = torch.tensor(x, device="cuda")
    c.neighbor_build(xd, torch.tensor(t, dtype=torch.int32, device="cuda"), box, 3.5)
    g = torch.full((table.size,), np.nan, dtype=torch.float64, device="cuda")
    c.backward(xd, torch.tensor([gE], dtype=torch.float64, device="cuda"), torch.tensor(gF, device="cuda"), None, g)
    torch.cuda.synchronize()
    c.close()
    assert scaled_err(table, g.cpu().numpy(), ref) <= 1e-10

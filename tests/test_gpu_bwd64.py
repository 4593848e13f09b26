"""The FP64 path's eight-lane parameter adjoint against the oracle's complex
step where its branches part: bonds at and beyond the sixteen kept ones, one and
two species, cutoffs that depend on the second record index, and lambda3 = 0
with m = 1 (whose derivative in lambda3 is not 0). Tolerance: 1e-10 of the
largest entry, each scaled by its parameter."""
import numpy as np
import pytest
import torch

import oracle
from tests import _systems as S
from tests.test_gpu_backward import scaled_err, weights
from tests.test_gpu_lanes64 import bcc, changed

pytestmark = pytest.mark.gpu
RC = 3.0


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1607_02904_gb300 as T
    T.load()
    return T


def cases():
    si = S.table_for(["Si"], oracle.mix_tersoff89)
    sic = S.table_for(["Si", "C"], oracle.mix_tersoff89)
    yield "bcc-14", *bcc(5, 2.9, 304), si
    yield "bcc-14-l3", *bcc(5, 2.9, 304), S.with_lambda3(si, 1.3, 3)
    yield "bcc-26", *bcc(5, 2.0, 305), si
    yield "si-l0m1", *S.si_cell(n=2, amp=0.15, seed=312), S.with_lambda3(si, 0.0, 1)
    yield "sic-cut-j", *S.sic_cell(n=2, sigma=0.12, seed=313), changed(
        sic, 10, lambda q, v: v - (0.05 if q in (1, 2, 5, 6) else 0.0))


CASES = list(cases())


@pytest.mark.parametrize("with_f", [True, False], ids=["forces", "energy"])
@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_against_complex_step(T, case, with_f):
    _, x, t, box, table = case
    gE, gF = weights(len(x), 92, with_f)
    nl = oracle.neighbors(x, box, RC)
    ref = np.zeros(table.size)
    for p in range(table.size):
        if p % oracle.NPAR:  # (not m)
            de, df = oracle.cs_param(x, t, box, table, nl, p)
            ref[p] = gE * de + (float((gF * df).sum()) if with_f else 0.0)
    ctx = T.Context(T.FP64)
    ctx.params(table)
    xd = torch.tensor(x, device="cuda")
    ctx.neighbor_build(xd, torch.tensor(t, dtype=torch.int32, device="cuda"), box, min(RC + 0.5, 0.5 * box.min()))
    g = torch.full((table.size,), np.nan, dtype=torch.float64, device="cuda")
    ctx.backward(xd, torch.tensor([gE], dtype=torch.float64, device="cuda"),
                 torch.tensor(gF, device="cuda") if with_f else None, None, g)
    got = g.cpu().numpy()
    ctx.close()
    assert np.isfinite(got).all() and np.all(got[::oracle.NPAR] == 0.0)
    assert scaled_err(table, got, ref) <= 1e-10

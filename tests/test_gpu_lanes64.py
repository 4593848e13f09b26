"""The FP64 path's lane-per-bond force kernel (4, 8 and 16 lanes per atom) against
the oracle: both table forms, bond counts at and beyond each lane count, cutoffs
that depend on the third record index, positions moved past the stored short
list's margin, images outside the box, and tables outside the integer formats
(which keep the per-thread kernel). Tolerance: the FP64 path's 1e-10."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from tests import _systems as S

pytestmark = pytest.mark.gpu
TOL = 1e-10
RC = 3.0


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1607_02904_gb300 as T
    T.load()
    return T


def bcc(n, a, seed):
    g = np.arange(n)
    base = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3).astype(np.float64)
    x = np.concatenate([base, base + 0.5]) * a
    box = np.full(3, n * a)
    rng = np.random.Generator(np.random.Philox(seed))
    return W.jitter_gaussian(x, 0.05, rng) % box, np.zeros(len(x), np.int32), box


def changed(table, field, fn):
    t = np.array(table).reshape(-1, 14).copy()
    for q in range(len(t)):
        t[q, field] = fn(q, t[q, field])
    return t.ravel()


def cases():
    si = S.table_for(["Si"], oracle.mix_tersoff89)
    sic = S.table_for(["Si", "C"], oracle.mix_tersoff89)
    x, t, box = S.si_cell(n=4, amp=0.2, seed=301)
    yield "si", x, t, box, si                                        # <= 4 bonds, some 5
    yield "si-l3m3", x, t, box, S.with_lambda3(si, 1.7322, 3)
    yield "si-l3m1", x, t, box, S.with_lambda3(si, 1.3, 1)
    yield "si-images", x + box * np.array([2, -1, 3]), t, box, si
    yield "si-wide-h", x, t, box, changed(si, 5, lambda q, v: 2.5)   # outside the formats
    yield "si-small-A", x, t, box, changed(si, 13, lambda q, v: 1e-9)
    x, t, box = S.sic_cell(n=4, sigma=0.12, seed=302)
    yield "sic", x, t, box, sic                                      # buckets of 8 and 16 lanes
    yield "sic-asym", x, t, box, changed(sic, 5, lambda q, v: v + 0.03 * q)
    # R of (i,j,k) differs from R of (i,k,k): f_C(r_ik) depends on j
    yield "sic-cut-j", x, t, box, changed(sic, 10, lambda q, v: v - (0.05 if q in (1, 2, 5, 6) else 0.0))
    x, t, box = S.packing_cell(n=400, seed=303)
    yield "packing-l3", x, t, box, S.with_lambda3(sic, 1.1, 3)
    x, t, box = bcc(5, 2.9, 304)                                     # 8 + 6 neighbours
    yield "bcc-14", x, t, box, si
    yield "bcc-14-l3", x, t, box, S.with_lambda3(si, 1.7322, 3)
    x, t, box = bcc(6, 2.0, 305)                                     # 26: beyond 16 lanes
    yield "bcc-26", x, t, box, si


CASES = list(cases())


@pytest.mark.parametrize("move", [0.0, 0.33], ids=["stored", "moved"])
@pytest.mark.parametrize("scatter", [0, 1], ids=["gather", "atomic"])
@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_against_oracle(T, case, scatter, move):
    _, x, t, box, table = case
    rng = np.random.Generator(np.random.Philox(306))
    y = x + rng.uniform(-1, 1, x.shape) * move / np.sqrt(3.0)
    w0 = y - box * np.floor(y / box)
    ref = oracle.compute(w0, t, box, table, oracle.neighbors(w0, box, RC))
    _, _, _, ea_ref = oracle.compute(w0, t, box, table, oracle.neighbors(w0, box, RC), eatom=True)
    ctx = T.Context(T.FP64)
    ctx.set_scatter(scatter)
    ctx.params(table)
    r_list = min(RC + 1.0, 0.5 * box.min())
    xd, yd = (torch.tensor(a, device="cuda") for a in (x, y))
    ctx.neighbor_build(xd, torch.tensor(t, dtype=torch.int32, device="cuda"), box, r_list)
    for _ in range(2):
        e = torch.zeros(1, dtype=torch.float64, device="cuda")
        f = torch.zeros_like(xd)
        w = torch.zeros(6, dtype=torch.float64, device="cuda")
        ea = torch.zeros(len(x), dtype=torch.float64, device="cuda")
        ctx.compute(yd, e, f, w)
        ctx.compute_peratom(yd, ea)
        f = f.cpu().numpy()
        assert abs(e.item() - ref[0]) <= TOL * abs(ref[0])
        assert np.abs(f - ref[1]).max() <= TOL * np.abs(ref[1]).max()
        assert np.abs(w.cpu().numpy() - ref[2]).max() <= TOL * np.abs(ref[2]).max()
        assert np.abs(ea.cpu().numpy() - ea_ref).max() <= TOL * np.abs(ea_ref).max()
    ctx.close()

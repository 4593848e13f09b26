"""Evaluations of the FP64 path on an existing list show positions that are not
finite and atoms at one place: the energy, the virial and the forces of the atoms
concerned are NaN, where fixed-point words would make them some finite place. Other
atoms' forces stay what they are. (A build refuses such positions.)"""
import numpy as np
import pytest
import torch

import oracle
from tests import _systems as S
from tests.test_gpu_lanes64 import bcc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1607_02904_gb300 as T
    T.load()
    return T


def systems():
    si = S.table_for(["Si"], oracle.mix_tersoff89)
    sic = S.table_for(["Si", "C"], oracle.mix_tersoff89)
    x, t, box = S.si_cell(n=4, amp=0.05, seed=601)
    yield "si", x, t, box, si                                    # four lanes
    yield "si-l3", x, t, box, S.with_lambda3(si, 1.3, 3)
    yield "sic", *S.sic_cell(n=5, sigma=0.1, seed=602), sic      # eight and sixteen lanes
    yield "bcc-14", *bcc(6, 2.9, 603), si
    yield "bcc-26", *bcc(6, 2.0, 604), si                        # the general path
    x, t, box = S.si_cell(n=4, amp=0.05, seed=605)
    yield "si-long", x, t, np.array([box[0], 5000.0, box[2]]), si


def bad_positions(x, box, what):
    y = x.copy()
    if what == "coincident":
        d = x - x[5]
        d -= box * np.round(d / box)
        r = (d * d).sum(1)
        r[5] = np.inf
        y[5] = x[int(r.argmin())]
    else:
        y[5, 1] = {"nan": np.nan, "inf": np.inf, "-inf": -np.inf}[what]
    return y


@pytest.mark.parametrize("scatter", [0, 1], ids=["gather", "atomic"])
@pytest.mark.parametrize("what", ["nan", "inf", "-inf", "coincident"])
@pytest.mark.parametrize("case", list(systems()), ids=lambda c: c[0])
def test_they_show(T, case, what, scatter):
    _, x, t, box, table = case
    r_list = min(4.0, 0.5 * box.min())
    ctx = T.Context(T.FP64)
    ctx.set_scatter(scatter)
    ctx.params(table)
    xd = torch.tensor(x, device="cuda")
    ctx.neighbor_build(xd, torch.tensor(t, dtype=torch.int32, device="cuda"), box, r_list)
    y = bad_positions(x, box, what)
    yd = torch.tensor(y, device="cuda")
    e = torch.zeros(1, dtype=torch.float64, device="cuda")
    f, w = torch.zeros_like(xd), torch.zeros(6, dtype=torch.float64, device="cuda")
    ea = torch.zeros(len(x), dtype=torch.float64, device="cuda")
    ctx.compute(yd, e, f, w)
    ctx.compute_peratom(yd, ea)
    f, ea = f.cpu().numpy(), ea.cpu().numpy()
    assert np.isnan(e.item()) and torch.isnan(w).all()
    assert np.isnan(f[5]).all() and np.isnan(ea[5])
    # the neighbours inside the cutoff at its old place; nothing beyond two list radii
    d = x - x[5]
    d -= box * np.round(d / box)
    r = np.sqrt((d * d).sum(1))
    near = (r < 2.6) & (np.arange(len(x)) != 5)
    if what != "coincident":
        assert near.any() and np.isnan(f[near]).all() and np.isnan(ea[near]).all()
    far = r > 2 * r_list + 2.0
    assert np.isfinite(f[far]).all() and np.isfinite(ea[far]).all()
    # and the context goes on with good positions
    e2, f2 = torch.zeros_like(e), torch.zeros_like(xd)
    ctx.compute(xd, e2, f2, None)
    ref = oracle.compute(x, t, box, table, oracle.neighbors(x, box, 3.0))
    assert abs(e2.item() - ref[0]) <= 1e-10 * abs(ref[0])
    assert np.abs(f2.cpu().numpy() - ref[1]).max() <= 1e-10 * np.abs(ref[1]).max()
    ctx.close()


def test_steps_without_rebuilds_show_them(T):
    x, t, box = S.si_cell(n=4, amp=0.05, seed=601)
    table = S.table_for(["Si"], oracle.mix_tersoff89)
    ctx = T.Context(T.FP64)
    ctx.params(table)
    xd = torch.tensor(x, device="cuda")
    ctx.neighbor_build(xd, torch.tensor(t, dtype=torch.int32, device="cuda"), box, 4.0)
    v, f = torch.zeros_like(xd), torch.zeros_like(xd)
    v[5, 0] = float("nan")
    th = torch.zeros((4, 3), dtype=torch.float64, device="cuda")
    ctx.md_step(xd, v, f, [28.0855], 0.001, 4, 0, th)
    assert torch.isnan(th[:, 0]).all()
    assert int(torch.isnan(f).any(1).sum()) >= 5
    ctx.close()


def test_batches_show_them_in_their_system_only(T):
    parts = [S.packing_cell(n=120, seed=611), S.packing_cell(n=90, seed=612)]
    x = np.concatenate([p[0] for p in parts])
    t = np.concatenate([p[1] for p in parts]).astype(np.int32)
    off = np.array([0, 120, 210], np.int32)
    boxes = np.stack([np.asarray(p[2], dtype=np.float64) * np.ones(3) for p in parts])
    batch = T.TersoffBatch(t, off, boxes, min(4.0, 0.5 * boxes.min()), T.FP64)
    table = torch.tensor(S.table_for(["Si", "C"], oracle.mix_tersoff89), dtype=torch.float64)
    e0, f0 = T.energy_forces(batch, torch.tensor(x, device="cuda"), table)
    y = x.copy()
    y[7, 2] = np.nan
    ctx = batch.ctx
    e, f = torch.zeros(2, dtype=torch.float64, device="cuda"), torch.zeros((210, 3), dtype=torch.float64, device="cuda")
    ctx.compute_batched(torch.tensor(y, device="cuda"), e, f, None)
    assert torch.isnan(e[0]) and torch.isnan(f[7]).all()
    assert abs(e[1] - e0[1]) <= 1e-13 * abs(e0[1])
    assert (f[120:] - f0[120:]).abs().max() <= 1e-12 * f0[120:].abs().max()


@pytest.mark.parametrize("scatter", [0, 1], ids=["gather", "atomic"])
@pytest.mark.parametrize("case", list(systems()), ids=lambda c: c[0])
def test_finite_forces_are_those_without_the_bad_position(T, case, scatter):
    # no atom is pushed by a term that has the bad position in it: its force is NaN or
    # what it is with all positions good (sums of the same terms: 1e-13 of the largest)
    _, x, t, box, table = case
    ctx = T.Context(T.FP64)
    ctx.set_scatter(scatter)
    ctx.params(table)
    xd = torch.tensor(x, device="cuda")
    ctx.neighbor_build(xd, torch.tensor(t, dtype=torch.int32, device="cuda"), box, min(4.0, 0.5 * box.min()))
    f0, f = torch.zeros_like(xd), torch.zeros_like(xd)
    ctx.compute(xd, None, f0, None)
    for at, axis, value in ((5, 0, np.nan), (17, 1, np.inf), (40, 2, -np.inf)):
        y = x.copy()
        y[at, axis] = value
        ctx.compute(torch.tensor(y, device="cuda"), None, f, None)
        good = torch.isfinite(f).all(1)
        assert not good[at]
        if good.any():
            assert (f[good] - f0[good]).abs().max() <= 1e-13 * f0.abs().max()
    ctx.close()

"""MD of small systems in the resident kernel against directly launched steps
(set_graphs(False)): the same device functions in the same order per atom, so
positions, velocities and forces agree bit for bit, and the thermo sums to
double rounding (their order over blocks is free). Sizes around the cluster's
16 blocks and the kernel's largest system; one to three species, lambda3;
rebuilds on the skin, by period, at every step, and never."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from tests import _systems as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1607_02904_gb300 as T
    T.load()
    return T


def system(cells, names, lam3=False, three=False):
    x, t, box = W.diamond(*cells, 5.432 if len(names) == 1 else 4.36, zincblende=len(names) > 1)
    table = S.table_for(names, oracle.mix_tersoff89)
    if three:  # a third species with the first one's records
        t2 = table.reshape(2, 2, 2, 14)
        pick = [0, 1, 0]
        table = np.array([[[t2[a, b, c] for c in pick] for b in pick] for a in pick]).ravel()
        t = np.where((t == 0) & (np.arange(len(t)) % 3 == 0), 2, t).astype(np.int32)
    if lam3:
        table = S.with_lambda3(table, 1.7322, 3)
    rng = np.random.Generator(np.random.Philox(411))
    x = W.jitter_gaussian(x, 0.04, rng)
    mass = [W.MASS_AMU["Si"], W.MASS_AMU["C"], W.MASS_AMU["Si"]][: 3 if three else len(names)]
    v = W.maxwell_velocities(t, np.array(mass), 900.0, rng)
    return x, v, t, box, table, mass


def steps(T, sysd, graphs, nsteps, every, thermo, calls=2):
    x, v, t, box, table, mass = sysd
    c = T.Context(T.MIXED)
    c.set_graphs(graphs)
    c.params(table)
    xd, vd = torch.tensor(x, device="cuda"), torch.tensor(v, device="cuda")
    c.neighbor_build(xd, torch.tensor(t, dtype=torch.int32, device="cuda"), box, 4.0)
    f = torch.zeros_like(xd)
    c.compute(xd, None, f)
    th = torch.zeros((nsteps, 3), dtype=torch.float64, device="cuda") if thermo else None
    rows, builds = [], []
    for _ in range(calls):
        c.md_step(xd, vd, f, mass, 0.001, nsteps, every, th)
        builds.append(c.md_rebuilds())
        if thermo:
            rows.append(th.cpu().numpy().copy())
    out = [a.cpu().numpy() for a in (xd, vd, f)]
    c.close()
    return out, rows, builds


@pytest.mark.parametrize("cells,names,lam3,three,nsteps,every,thermo", [
    ((2, 2, 2), ["Si"], False, False, 60, -1, True),     # 64 atoms: one block
    ((3, 3, 3), ["Si"], True, False, 40, -1, False),
    ((8, 8, 4), ["Si"], False, False, 60, -1, True),     # 2,048: sixteen blocks
    ((8, 8, 4), ["Si"], False, False, 25, 1, True),      # a rebuild at every step
    ((3, 3, 29), ["Si"], False, False, 60, -1, True),    # 2,088: seventeen blocks
    ((3, 3, 29), ["Si"], False, False, 23, 10, False),   # the period carries over calls
    ((3, 4, 5), ["Si"], False, False, 30, 0, True),      # never
    ((16, 16, 32), ["Si"], False, False, 40, -1, True),  # 65,536: the largest
    ((16, 16, 33), ["Si"], False, False, 12, 5, True),   # one beyond: graph launches
    ((2, 2, 2), ["Si", "C"], False, False, 30, -1, True),
    ((4, 4, 5), ["Si", "C"], True, False, 20, 7, True),
    ((3, 3, 3), ["Si", "C"], False, True, 20, 7, True),
])
def test_equals_direct_launches(T, cells, names, lam3, three, nsteps, every, thermo):
    sysd = system(cells, names, lam3, three)
    a, ra, ba = steps(T, sysd, True, nsteps, every, thermo)
    b, rb, bb = steps(T, sysd, False, nsteps, every, thermo)
    assert ba == bb
    for p, q in zip(a, b):
        assert np.array_equal(p, q)
    for p, q in zip(ra, rb):
        assert np.abs(p - q).max() <= 1e-12 * np.abs(q).max()


def test_long_call_crosses_launch_bound(T):
    # more steps than one launch takes, without and with a period
    sysd = system((2, 2, 2), ["Si"])
    for every in (0, 4099):
        x, v = sysd[0], 0.02 * sysd[1]
        a, _, _ = steps(T, (x, v) + sysd[2:], True, 4200, every, False, calls=1)
        b, _, _ = steps(T, (x, v) + sysd[2:], False, 4200, every, False, calls=1)
        for p, q in zip(a, b):
            assert np.array_equal(p, q)


def test_overflow_inside_the_call_reruns(T):
    # the list's capacity is exceeded by a rebuild inside the call: the start
    # state is restored and the steps run again with grown lists
    x, v, t, box, table, mass = system((3, 3, 3), ["Si"])
    outs = []
    for graphs in (True, False):
        c = T.Context(T.MIXED)
        c.set_graphs(graphs)
        c.params(table)
        xd, vd = torch.tensor(x, device="cuda"), torch.tensor(v, device="cuda")
        td = torch.tensor(t, dtype=torch.int32, device="cuda")
        c.set_neighbor_capacity(1)
        c.neighbor_build(xd, td, box, 3.85)
        cap, most = c.neighbor_capacity()
        c.set_neighbor_capacity(most)  # no room to spare
        c.neighbor_build(xd, td, box, 3.85)
        f = torch.zeros_like(xd)
        c.compute(xd, None, f)
        c.md_step(xd, vd, f, mass, 0.001, 60, 5)
        outs.append([a.cpu().numpy() for a in (xd, vd, f)] + [c.neighbor_capacity()[0]])
        c.close()
    assert outs[0][3] > most and outs[1][3] > most
    for p, q in zip(outs[0][:3], outs[1][:3]):
        # the rerun's lists have another capacity, not another order
        assert np.array_equal(p, q)

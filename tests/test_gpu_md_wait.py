"""A wait of the resident MD kernel that runs out: the call restores its start, runs
its steps by launches and succeeds; later calls take launches too. The limit is one
poll, so that of the blocks of a step all but the last to arrive give up at once,
while the last ones go on: partly done steps, forces in the fallback buffer.

Bound on the differences from direct launches: past the short list's margin forces
are summed by FP64 atomics in any order, 2^-53 of each of some twenty terms, which
sixty steps carry on: 1e-12 of the largest value."""
import numpy as np
import pytest
import torch

import oracle
from tests import _systems as S
from tests.test_gpu_resident import system

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1607_02904_gb300 as T
    T.load()
    return T


def context(T, sysd, move=0.0):
    x, v, t, box, table, mass = sysd
    c = T.Context(T.MIXED)
    c.params(table)
    xd, vd = torch.tensor(x, device="cuda"), torch.tensor(v, device="cuda")
    c.neighbor_build(xd, torch.tensor(t, dtype=torch.int32, device="cuda"), box, 4.0)
    if move:
        rng = np.random.Generator(np.random.Philox(801))
        xd += torch.tensor(rng.uniform(-1, 1, x.shape) * move / np.sqrt(3.0), device="cuda")
    f = torch.zeros_like(xd)
    c.compute(xd, None, f)
    return c, xd, vd, f, mass


@pytest.mark.parametrize("cells,names", [((3, 3, 29), ["Si"]), ((8, 8, 8), ["Si", "C"]), ((16, 16, 32), ["Si"])],
                         ids=["17-blocks", "sic-32-blocks", "512-blocks"])
@pytest.mark.parametrize("every,nsteps", [(-1, 30), (0, 12), (7, 30), (5, 20)])
def test_the_call_runs_by_launches(T, cells, names, every, nsteps):
    sysd = system(cells, names)
    res, launches = [], []
    for limited in (False, True):
        c, xd, vd, f, mass = context(T, sysd)
        if limited:
            c.set_md_wait_limit(1)
        else:
            c.set_graphs(False)
        th = torch.zeros((nsteps, 3), dtype=torch.float64, device="cuda")
        for _ in range(2):
            l0 = c.launch_count()
            c.md_step(xd, vd, f, mass, 0.001, nsteps, every, th)
            launches.append(c.launch_count() - l0)
        res.append([a.cpu().numpy() for a in (xd, vd, f, th)])
        c.close()
    assert min(launches) >= 2 * nsteps  # no call stayed in the resident kernel
    for a, b in zip(*res):
        assert np.abs(a - b).max() <= 1e-12 * np.abs(a).max()


def test_nothing_is_left_behind(T):
    # steps past the short list's margin scatter into the fallback buffer; forces on an
    # expired list read it afterwards
    sysd = system((8, 8, 8), ["Si"])
    x, v, t, box, table, mass = sysd
    for _ in range(5):
        c, xd, vd, f, mass = context(T, sysd, move=0.33)
        c.set_md_wait_limit(1)
        start = [a.clone() for a in (xd, vd, f)]
        c.md_step(xd, vd, f, mass, 0.001, 5, 0)
        ref, *rest = context(T, sysd, move=0.33)
        ref.set_graphs(False)
        ref.md_step(*start, mass, 0.001, 5, 0)
        # (the rerun has a list of its own start: sums in another order, in float)
        assert (xd - start[0]).abs().max() <= 1e-7 and (vd - start[1]).abs().max() <= 1e-4
        rng = np.random.Generator(np.random.Philox(802))
        yd = xd + torch.tensor(rng.uniform(-1, 1, x.shape) * 0.33 / np.sqrt(3.0), device="cuda")
        for _ in range(2):
            c.compute(yd, None, f)
            y = yd.cpu().numpy()
            y = y - box * np.floor(y / box)
            want = oracle.compute(y, t, box, table, oracle.neighbors(y, box, 3.0))[1]
            assert np.abs(f.cpu().numpy() - want).max() <= 2e-5 * np.abs(want).max()
        c.close()
        ref.close()


def test_limits_are_checked(T):
    c = T.Context(T.MIXED)
    for bad in (0, (1 << 22) + 1):
        with pytest.raises(Exception):
            c.set_md_wait_limit(bad)
    c.set_md_wait_limit(1 << 22)
    c.close()

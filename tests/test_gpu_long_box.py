"""The FP64 path in long boxes: a cluster in a vacuum box of any length has the
forces, energy, steps and gradients that it has in a short one.

Positions are rounded to 2^-(fix64 + 1) A, at most 2^-52 up to edges of 2^17 A: a
bond vector is off by 2^-51, and a force by that times its stiffness, some 50 eV/A^2
for each of four bonds: 1e-13 eV/A, 3e-14 of the largest forces here (3 to 5 eV/A).
Beyond 2^17 A the bound grows with the edge.
Edges are whole numbers and positions multiples of 2^-30 A, exact in doubles at
every place of the box."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from tests import _systems as S

pytestmark = pytest.mark.gpu
TOL = 3e-14
SHORT = 64.0


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1607_02904_gb300 as T
    T.load()
    return T


def cluster(names):
    x, t, _ = S.si_cell(n=3, amp=0.2, seed=501) if len(names) == 1 else S.sic_cell(n=3, sigma=0.1, seed=502)
    return np.round(x * 2.0 ** 30) / 2.0 ** 30, t, S.table_for(names, oracle.mix_tersoff89)


def context(T, x, t, box, table):
    ctx = T.Context(T.FP64)
    ctx.params(table)
    xd = torch.tensor(x, device="cuda")
    ctx.neighbor_build(xd, torch.tensor(t, dtype=torch.int32, device="cuda"), np.asarray(box, dtype=np.float64), 4.0)
    return ctx, xd


def evaluate(T, x, t, box, table, moved=None):
    ctx, xd = context(T, x, t, box, table)
    if moved is not None:
        xd = torch.tensor(moved, device="cuda")
    e = torch.zeros(1, dtype=torch.float64, device="cuda")
    f = torch.zeros_like(xd)
    w = torch.zeros(6, dtype=torch.float64, device="cuda")
    ctx.compute(xd, e, f, w)
    ctx.close()
    return e.item(), f.cpu().numpy(), w.cpu().numpy()


def close(a, b, tol=TOL):
    a, b = np.atleast_1d(a), np.atleast_1d(b)
    return np.abs(a - b).max() <= tol * np.abs(b).max()


EDGES = [1000.0, 2048.0, 2049.0, 5000.0, 100000.0, 1048576.0]


@pytest.mark.parametrize("names", [["Si"], ["Si", "C"]], ids=["si", "sic"])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("edge", EDGES)
def test_forces_as_in_a_short_box(T, edge, axis, names):
    x, t, table = cluster(names)
    ref = evaluate(T, x, t, [SHORT] * 3, table)
    box = [SHORT] * 3
    box[axis] = edge
    for at in (0.0, -7.0, 3 * edge + 1.0, -2 * edge - 5.0):  # at the origin, over the edge, images
        y = x.copy()
        y[:, axis] += at
        got = evaluate(T, y, t, box, table)
        tol = TOL * max(1.0, edge / 2.0 ** 17)
        assert close(got[0], ref[0], tol) and close(got[1], ref[1], tol) and close(got[2], ref[2], tol)


def test_two_clusters_far_apart_and_all_axes_long(T):
    x, t, table = cluster(["Si"])
    e, f, w = evaluate(T, x, t, [SHORT] * 3, table)
    box = [60000.0, 8192.0 * 3, 70000.0]
    for shift in ((8192.0, 0, 0), (30000.0, 16384.0, 35000.0), (59900.0, 24500.0, 69900.0)):
        got = evaluate(T, np.concatenate([x, x + np.array(shift)]), np.concatenate([t, t]), box, table)
        assert close(got[0], 2 * e) and close(got[1][:len(x)], f) and close(got[1][len(x):], f)


def test_an_atom_moved_by_the_words_range_is_far(T):
    # 2^64 units of 2^-51 A: the difference words repeat, the coarse words do not
    x, t, table = cluster(["Si"])
    box = [100000.0, SHORT, SHORT]
    out = []
    for far in (8000.0, 8192.0, 2 * 8192.0, 100000.0 - 8192.0):
        y = x.copy()
        y[5, 0] += far
        out.append(evaluate(T, x, t, box, table, moved=y))
    for got in out[1:]:  # (past the short list's margin: sums by atomics)
        assert close(got[0], out[0][0]) and close(got[1], out[0][1])
    assert np.all(out[0][1][5] == 0.0)


def test_steps_gradients_and_batches_as_in_a_short_box(T):
    x, t, table = cluster(["Si", "C"])
    v0 = W.maxwell_velocities(t, np.array([28.0855, 12.011]), 600.0, np.random.Generator(np.random.Philox(503)))
    rng = np.random.Generator(np.random.Philox(504))
    gE = torch.tensor([0.6], dtype=torch.float64, device="cuda")
    gF = torch.tensor(rng.standard_normal(x.shape), device="cuda")
    res = []
    for box in ([SHORT] * 3, [SHORT, 100000.0, 3000.0]):
        ctx, xd = context(T, x, t, box, table)
        g = torch.zeros(table.size, dtype=torch.float64, device="cuda")
        gx = torch.zeros_like(xd)
        ctx.backward(xd, gE, gF, gx, g)
        v, f = torch.tensor(v0, device="cuda"), torch.zeros_like(xd)
        ctx.compute(xd, None, f)
        ctx.md_step(xd, v, f, [28.0855, 12.011], 0.0005, 12, 5)
        res.append([a.cpu().numpy() for a in (g, gx, xd, v, f)])
        ctx.close()
    for a, b in zip(*res):
        assert close(b, a, 20 * TOL)  # (second derivatives, and twelve steps of exponential growth)
    off = np.array([0, len(x), 2 * len(x)], np.int32)
    batch = T.TersoffBatch(np.concatenate([t, t]).astype(np.int32), off, np.array([[100000.0, 900.0, 3000.0], [SHORT] * 3]), 4.0, T.FP64)
    e, f = T.energy_forces(batch, torch.tensor(np.concatenate([x, x]), device="cuda"), torch.tensor(table, dtype=torch.float64))
    e, f = e.cpu().numpy(), f.cpu().numpy()
    ref = evaluate(T, x, t, [SHORT] * 3, table)
    for k in (0, 1):
        assert close(e[k], ref[0]) and close(f[k * len(x):(k + 1) * len(x)], ref[1])

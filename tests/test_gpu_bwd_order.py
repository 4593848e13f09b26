"""The mixed path's table gradient does not depend on which atoms share a warp.
Their order comes from atomics and differs between contexts; an atom's own terms
are summed in float in the order of its list, sums over atoms in float pairs and
double. Sizes: one sorting block, several warps and blocks, a large crystal, a
batch of uneven cells.

Tolerance: a plain float sum over a warp moves the gradient by up to 1e-7 of its
norm, some 2 units of 2^-24; pairs carry twice the bits, 2 units of 2^-47, and
block totals in double less: 1e-12 of the norm leaves a factor of 70."""
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


def crystal(cells, names, sigma):
    x, t, box = W.diamond(*cells, 5.432 if len(names) == 1 else 4.36, zincblende=len(names) > 1)
    return W.jitter_gaussian(x, sigma, np.random.Generator(np.random.Philox(77))), t, box


@pytest.mark.parametrize("cells,names,sigma,repeats", [
    ((3, 3, 3), ["Si"], 0.05, 12), ((7, 6, 9), ["Si"], 0.15, 8), ((9, 8, 7), ["Si", "C"], 0.12, 8),
    ((33, 32, 33), ["Si"], 0.1, 3),
], ids=["216", "3024", "sic-4032", "278784"])
def test_fresh_contexts_agree(T, cells, names, sigma, repeats):
    x, t, box = crystal(cells, names, sigma)
    table = S.table_for(names, oracle.mix_tersoff89)
    xd, td = torch.tensor(x, device="cuda"), torch.tensor(t, dtype=torch.int32, device="cuda")
    gE = torch.tensor([0.7], dtype=torch.float64, device="cuda")
    gF = torch.tensor(np.random.Generator(np.random.Philox(78)).standard_normal(x.shape), device="cuda")
    got = []
    for _ in range(repeats):
        ctx = T.Context(T.MIXED)
        ctx.params(table)
        ctx.neighbor_build(xd, td, box, 4.0)
        g = torch.zeros(table.size, dtype=torch.float64, device="cuda")
        ctx.backward(xd, gE, gF, None, g)
        got.append(g.cpu().numpy())
        ctx.close()
    assert np.linalg.norm(got[0]) > 0
    for g in got[1:]:
        assert np.linalg.norm(g - got[0]) <= 1e-12 * np.linalg.norm(got[0])


def test_fresh_batches_agree(T):
    parts = [S.packing_cell(n=n, seed=60 + n) for n in (64, 200, 333, 97)]
    x = np.concatenate([p[0] for p in parts])
    t = np.concatenate([p[1] for p in parts])
    off = np.concatenate([[0], np.cumsum([len(p[0]) for p in parts])]).astype(np.int32)
    boxes = np.stack([np.asarray(p[2], dtype=np.float64) * np.ones(3) for p in parts])
    r_list = min(4.0, 0.5 * boxes.min())
    table = S.table_for(["Si", "C"], oracle.mix_tersoff89)
    got = []
    for _ in range(8):
        b = T.TersoffBatch(t.astype(np.int32), off, boxes, r_list, T.MIXED)
        tb = torch.tensor(table, dtype=torch.float64, requires_grad=True)
        xd = torch.tensor(x, device="cuda")
        e, f = T.energy_forces(b, xd, tb)
        loss = (e * torch.arange(1, len(parts) + 1, device="cuda")).sum() + (f * torch.sin(17.0 * xd)).sum()
        got.append(torch.autograd.grad(loss, [tb])[0].numpy())
    for g in got[1:]:
        assert np.linalg.norm(g - got[0]) <= 1e-12 * np.linalg.norm(got[0])


@pytest.mark.parametrize("names", [["Si"], ["Si", "C"]], ids=["si", "sic"])
def test_infinite_sums_stay_infinite(T, names):
    # an infinite energy weight: the A entries' terms are all +inf, the B entries' -inf
    x, t, box = crystal((3, 3, 3), names, 0.05)
    table = S.table_for(names, oracle.mix_tersoff89)
    ctx = T.Context(T.MIXED)
    ctx.params(table)
    xd = torch.tensor(x, device="cuda")
    ctx.neighbor_build(xd, torch.tensor(t, dtype=torch.int32, device="cuda"), box, 4.0)
    g = torch.zeros(table.size, dtype=torch.float64, device="cuda")
    ctx.backward(xd, torch.tensor([np.inf], dtype=torch.float64, device="cuda"), None, None, g)
    g = g.cpu().numpy().reshape(-1, 14)
    ctx.close()
    ns = len(names)
    for a in range(ns):
        for b in range(ns):
            if ns == 2 and a == b:
                continue  # (no bonds between like atoms in zincblende)
            r = g[(a * ns + b) * ns + b]
            assert r[13] == np.inf and r[9] == -np.inf

"""The warp-per-atom list build of small systems where a cell holds more atoms
than a warp has lanes, and with odd counts, against the oracle's lists (exact)."""
import numpy as np
import pytest
import torch

import oracle
from tests import _systems as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,length,r_list,seed", [
    (432, 12.0, 6.0, 601),   # 54 atoms per cell
    (431, 12.0, 3.9, 602),
    (33, 9.0, 3.1, 603),
    (1, 12.0, 4.0, 604),
])
def test_full_cells_match_oracle(n, length, r_list, seed):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1607_02904_gb300 as T
    T.load()
    rng = np.random.Generator(np.random.Philox(seed))
    box = np.array([length, length, length])
    x = rng.uniform(0.0, length, (n, 3))
    c = T.Context(T.MIXED)
    c.params(S.table_for(["Si"], oracle.mix_tersoff89))
    c.neighbor_build(torch.tensor(x, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda"), box, r_list)
    ref_cnt, ref = oracle.neighbors(x, box, r_list, cap=512)
    cnt, nbr, st = c.neighbor_export(512)
    cnt, nbr = cnt.cpu().numpy(), nbr.cpu().numpy()
    c.close()
    assert st == 0
    assert np.array_equal(cnt, ref_cnt)
    for i in range(n):
        assert np.array_equal(nbr[i, : cnt[i]], ref[i, : cnt[i]])

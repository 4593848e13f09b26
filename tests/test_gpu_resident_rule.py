"""Which MD calls of small systems run in the resident kernel, seen by the launches
they enqueue: calls of whole rebuild periods only while one cluster holds the system
(16 blocks of 128 atoms; a replayed graph of launches is faster beyond), the others
up to 65,536 atoms."""
import pytest
import torch

from tests.test_gpu_md_wait import context
from tests.test_gpu_resident import system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cells,every,nsteps,resident", [
    ((8, 8, 4), 10, 40, True),      # 2,048 atoms: the largest cluster
    ((3, 3, 29), 10, 40, False),    # 2,088
    ((3, 3, 29), 10, 25, True),     # not whole periods
    ((3, 3, 29), -1, 40, True),
    ((3, 3, 29), 0, 40, True),
    ((16, 16, 32), 20, 40, False),  # 65,536
    ((16, 16, 32), -1, 40, True),
    ((16, 16, 33), -1, 40, False),
])
def test_rule(cells, every, nsteps, resident):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1607_02904_gb300 as T
    T.load()
    c, xd, vd, f, mass = context(T, system(cells, ["Si"]))
    for _ in range(2):
        l0 = c.launch_count()
        c.md_step(xd, vd, f, mass, 0.001, nsteps, every)
        # by launches two a step; resident one a stretch, and some eight per rebuild
        launches = c.launch_count() - l0 - 10 * c.md_rebuilds()
        assert (launches < nsteps) == resident
    c.close()

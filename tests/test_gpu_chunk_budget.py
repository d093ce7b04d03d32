"""Grid points per Alg. 6 chunk where G_I^YZ is rebuilt and the memory budget allows
fewer than 16 of them (needs a GB300).

P = 6000: one grid point of G takes P^2 words = 288 MB and the budget of a chunk
with a stated workspace limit is 4 GiB, so 14 points.  From 512 grid points on the
float-pair triangle has sums with bounds per 16 points; they must not raise the
chunk above the budget.  Two contexts that differ in the number of grid points
(500 and 520) only: the second one's larger arrays are U (o G P words, 1.9 MB more)
and what is made of x and z; two grid points of G more would be 576 MB."""
import numpy as np
import pytest
import torch

from synth import make_system
from tests.gpu_util import context

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()


def _held(G):
    """Device bytes of a context with G grid points."""
    s = make_system(2, 3, 24, G, 4, 1)
    P = 6000
    s.Y = np.random.default_rng(2).standard_normal((5, P)) / P ** 0.5
    free = torch.cuda.mem_get_info()[0]
    with context(s, precision=2, t2sq_route=1, x_block6=8, workspace_bytes=64 << 30) as ctx:
        torch.cuda.synchronize()
        return free - torch.cuda.mem_get_info()[0]


def test_chunk_of_rebuilt_g_stays_within_its_budget():
    _held(500)      # what the library holds besides contexts is there now
    a, b = _held(500), _held(520)
    print(f"device memory of the contexts: {a / 1e9:.2f} and {b / 1e9:.2f} GB")
    assert b - a < 288e6

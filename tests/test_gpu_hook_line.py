"""The line between hooking all edges in one launch and in slices (m^2 = 490000 n): random graphs with a
little fewer and a little more edges than that, on both sides of the larger first slice's limit, against the
oracle."""

import math

import pytest

import oracle
import synth
from _gpu_util import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [5, 1025, 16385, 70001, 1 << 18, (1 << 18) + 1])
@pytest.mark.parametrize("over", [-1, 0, 1, 300])
def test_either_side(n, over):
    import paper_2103_15217_gb300 as etl
    m = math.isqrt(490000 * n) + over
    e = synth.easy_graph(n, m, seed=n)
    st = etl.new_status()
    got = host(etl.find_bridges(dev(e), n, status=st))
    assert int(st) == 0
    assert (got == oracle.bridges_dfs(n, e)).all()

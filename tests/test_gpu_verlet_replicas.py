"""Verlet-skin lists of periodic replicas whose boxes are large enough for
cells (three or more of rc + skin per edge): the candidate rows come from the
cells of every replica, in every rebuild, and the filtered pairs are the
oracle's."""
import pytest

from paper_2510_06562_gb300 import inputs as I
from test_gpu_verlet import _check_pairs, _ctx, _displace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_side,n_rep", [(6, 2), (6, 5), (8, 3)])
def test_cells_of_every_replica(n_side, n_rep):
    s = I.replicas([I.make_water(n_side, round(3.105 * n_side, 2), 10 + k) for k in range(n_rep)])
    with _ctx(s, 1.0) as ctx:
        for seed in range(3):
            ctx.set_state(s.x if seed == 0 else _displace(s.x, 1.5, seed))
            _check_pairs(ctx, s, ctx.get_state()[0])
        assert ctx.neighbor_stats()[1] == 3                    # every state rebuilt the candidate rows

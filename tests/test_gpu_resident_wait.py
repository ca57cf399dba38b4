"""A wait of the resident PCG kernel that runs out ends the launch: every thread block
leaves, and the context solves as before afterwards.  The wait is taken as run out by the
host's request in one block of the problem's group (it ends as usual itself); in a
cooperative launch the others then wait for that block until their own limit."""
import numpy as np
import pytest

from synth import bar_twist_config, figure_config

pytestmark = pytest.mark.gpu

CASES = [
    ("bar", dict(precision="fp64"), 3),          # one cluster, one unit a block
    ("fig30000", dict(precision="mixed"), 0),    # one cluster, blocks with one and with two coarse units
    ("fig30000", dict(precision="mixed"), 7),
    ("fig60000", dict(precision="mixed"), 5),    # cooperative launch
]


def config(name):
    if name == "bar":
        return bar_twist_config()
    return figure_config(int(name[3:]), model="corot", seeds=[3])


@pytest.mark.parametrize("name,opts,iteration", CASES)
def test_launch_ends_when_a_wait_runs_out(name, opts, iteration):
    from paper_2408_04066_gb300 import mfem
    cfg = config(name)
    xf = np.asarray(cfg["xfs"])[:1]
    ctx = mfem.Context.from_config(cfg, tile_rows=128, spmv_split=1, **opts)
    ref, st0 = ctx.solve_batch(xf)
    ctx.expire_wait(iteration)
    try:
        ctx.solve_batch(xf)
    except mfem.MfemError as e:
        assert e.status in (mfem.MFEM_ECUDA, mfem.MFEM_ETIMEOUT)
    for _ in range(2):
        x, st = ctx.solve_batch(xf)
        assert np.array_equal(x, ref) and st[0]["pcg_iters"] == st0[0]["pcg_iters"]
    ctx.close()

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


SAME = [
    # config, model, options, iteration: the result is the undisturbed solve's, bit for bit
    ("bar", "arap", dict(precision="fp64"), 2),                             # FP64, cluster
    ("fig3000", "snh", dict(precision="mixed"), 4),                         # the predictor step is cut short
    ("fig3000", "snh", dict(precision="mixed", precond="block_jacobi"), 9),  # no coarse product: only the block's own word
    ("fig30000", "snh", dict(precision="mixed", rotation="polar"), 1),
    ("fig60000", "snh", dict(precision="mixed"), 6),                        # cooperative launch
    ("fig60000", "corot", dict(precision="fp64", cg_max=9000), 6),          # ... of limited length, read before the step
]


@pytest.mark.parametrize("name,model,opts,iteration", SAME)
def test_cut_short_solve_is_done_again(name, model, opts, iteration):
    from paper_2408_04066_gb300 import mfem
    cfg = dict(config(name), model=model)
    xf = np.concatenate([np.asarray(cfg["xfs"])] * 2)[:2]
    ctx = mfem.Context.from_config(cfg, tile_rows=128, spmv_split=1, max_batch=2, **opts)
    ref, st0 = ctx.solve_batch(xf)
    ctx.expire_wait(iteration)
    x, st = ctx.solve_batch(xf)
    p = ctx.profile()
    assert p["kernel_launches"] > p["pcg_launches"]          # launches per iteration: streamed
    assert np.array_equal(x, ref)
    for a, b in zip(st, st0):
        for k in ("status", "newton_iters", "pcg_iters", "converged", "energy", "rel_grad"):
            assert a[k] == b[k], k
    ctx.close()


def test_cut_short_warm_stream():
    """A warm-started stream whose predictor step, and later whose Newton step, is cut short
    carries the same state from frame to frame."""
    from paper_2408_04066_gb300 import mfem
    from synth import figure_animation
    cfg = dict(config("fig3000"), model="snh")
    anim = figure_animation(cfg["joints"], cfg["parent"], 7, 5)
    runs = []
    for disturbed in (False, True):
        ctx = mfem.Context.from_config(cfg, init="warm", tile_rows=128, spmv_split=1, max_batch=1)
        got = []
        for f in range(5):
            if disturbed and f in (1, 3):
                ctx.expire_wait(0 if f == 1 else 12)
            x, st = ctx.solve_batch(anim[f][None])
            got.append((x, st[0]["newton_iters"], st[0]["pcg_iters"]))
        runs.append(got)
        ctx.close()
    for (xa, na, pa), (xb, nb, pb) in zip(*runs):
        assert np.array_equal(xa, xb) and (na, pa) == (nb, pb)


def test_cut_short_served_request():
    from paper_2408_04066_gb300 import mfem
    cfg = dict(config("fig30000"), model="snh")
    opts = dict(tile_rows=256, spmv_split=1)
    ctx = mfem.Context.from_config(cfg, **opts)
    ref = ctx.solve_batch(np.asarray(cfg["xfs"])[:1])
    ctx.close()
    srv = mfem.Server(max_slots=2)
    ctx = mfem.Context.from_config(cfg, **opts)
    ctx.expire_wait(5)
    mid = srv.add(ctx)
    for _ in range(2):
        x, st, _ = srv.wait(srv.submit(mid, cfg["xfs"][0]))
        assert np.array_equal(x, ref[0][0])
        assert (st["newton_iters"], st["pcg_iters"]) == (ref[1][0]["newton_iters"], ref[1][0]["pcg_iters"])
    srv.close()


def test_cut_short_at_any_iteration():
    """One cluster of which a block without coarse units tells the others, at every iteration of
    the first solve: it may run ahead of blocks that have not yet left the barrier before."""
    from paper_2408_04066_gb300 import mfem
    cfg = dict(config("fig3000"), model="corot")
    xf = np.asarray(cfg["xfs"])[:1]
    ref = None
    for iteration in range(-1, 16):
        ctx = mfem.Context.from_config(cfg, tile_rows=128, spmv_split=1, max_batch=1)
        ctx.expire_wait(iteration)
        x, st = ctx.solve_batch(xf)
        if ref is None:
            ref, st0 = x, st
        assert np.array_equal(x, ref) and st[0]["pcg_iters"] == st0[0]["pcg_iters"], iteration
        ctx.close()

"""The resident PCG kernel's further routes against the streamed kernels, bit for bit: five
to eight units of 64 rows a block in both precisions, the shared-memory ring of the coarse
inverse kept (200k tets) and streamed (a block with two coarse units: 300k), aggregates of
two units (345k), two problems on the chip, more clusters than run at once, blocks without
rows (9 to 15 units on 16 blocks), and meshes of unlike size in one launch."""
import functools

import numpy as np
import pytest

from synth import figure_config

pytestmark = pytest.mark.gpu


@functools.lru_cache(maxsize=2)
def config(tets):
    return dict(figure_config(tets, seeds=[3, 4]), model="corot")


def resident(ctx):
    p = ctx.profile()
    return 2 * p["kernel_launches"] < p["pcg_launches"]


CASES = [
    # tets, batches that fit, one that does not, options
    (2300, (1, 8), 80, dict(precision="mixed")),
    (2300, (1, 8), 80, dict(precision="fp64")),
    (20000, (1, 12), 24, dict(precision="mixed")),
    (30000, (1, 8), 24, dict(precision="fp64")),
    (150000, (1, 2), 4, dict(precision="mixed")),
    (200000, (1,), 2, dict(precision="mixed")),
    (200000, (1,), 2, dict(precision="fp64")),
    (300000, (1,), 2, dict(precision="mixed")),
    (300000, (1,), 2, dict(precision="fp64")),
    (345000, (1,), 2, dict(precision="mixed")),
    (345000, (1,), 2, dict(precision="mixed", precond="block_jacobi")),
]


@pytest.mark.parametrize("tets,few,many,opts", CASES)
def test_resident_equals_streamed(tets, few, many, opts):
    from paper_2408_04066_gb300 import mfem
    cfg = config(tets)
    xf = np.asarray(cfg["xfs"])
    batch = lambda b: np.concatenate([xf] * (-(-b // 2)))[:b]  # noqa: E731
    ctx = mfem.Context.from_config(cfg, max_batch=many, newton_max=3, tile_rows=128, **opts)
    ref, st0 = ctx.solve_batch(batch(many))
    p = ctx.profile()   # mostly streamed: the last pose of a batch may end alone in the resident kernel
    assert 2 * p["kernel_launches"] > p["pcg_launches"]
    for b in few:
        x, st = ctx.solve_batch(batch(b))
        assert resident(ctx)
        for i in range(b):
            assert np.array_equal(x[i], ref[i]), (b, i)
            assert st[i]["pcg_iters"] == st0[i]["pcg_iters"] and st[i]["newton_iters"] == st0[i]["newton_iters"]
    ctx.close()


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_unlike_meshes_in_one_launch(precision):
    from paper_2408_04066_gb300 import mfem
    cfgs = [config(1500), config(250000)]
    opts = dict(precision=precision, tile_rows=128, newton_max=3, max_batch=2)
    ctxs = [mfem.Context.from_config(c, **opts) for c in cfgs]
    xfs = [np.asarray(cfgs[0]["xfs"]), np.asarray(cfgs[1]["xfs"])[:1]]
    outs, stats = mfem.solve_multi(ctxs, xfs)
    assert resident(ctxs[0])
    for c, x, o, ss in zip(ctxs, xfs, outs, stats):
        for b in range(len(x)):
            ref, st = c.solve_batch(x[b:b + 1])
            assert np.array_equal(ref[0], o[b]) and st[0]["pcg_iters"] == ss[b]["pcg_iters"]
        c.close()

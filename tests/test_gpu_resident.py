"""The resident PCG kernel (problems that fit the chip: one launch runs a whole
solve) against the streamed kernels: a pose alone takes the first, the same pose
in a batch too large for the chip the second, and both do the same arithmetic in
the same order, so positions and iteration counts are equal bit for bit.  Sizes:
one to many 64-row units a CTA, ragged last units, clusters and the cooperative
launch, both precisions (FP64: every reduction tile), with and without the coarse
space, aggregates of several units."""
import numpy as np
import pytest

from synth import bar_twist_config, figure_config

pytestmark = pytest.mark.gpu

CASES = [
    # config, batch that does not fit, options
    ("bar", 160, dict(precision="mixed")),
    ("bar", 160, dict(precision="fp64", tile_rows=64)),
    ("bar", 160, dict(precision="fp64", tile_rows=128)),
    ("bar", 160, dict(precision="mixed", precond="block_jacobi")),
    ("fig3000", 80, dict(precision="mixed", coarse_agg=256)),
    ("fig3000", 80, dict(precision="fp64", tile_rows=256)),
    ("fig10000", 32, dict(precision="mixed", constraint="penalty", k_s=1e5)),
    ("fig50000", 8, dict(precision="mixed")),
    ("fig50000", 8, dict(precision="mixed", precond="block_jacobi", coarse_agg=0)),
    ("fig50000", 8, dict(precision="fp64", tile_rows=128, coarse_agg=128)),
]


def config(name):
    if name == "bar":
        return bar_twist_config()
    return figure_config(int(name[3:]), model="snh" if name != "fig10000" else "corot", seeds=[3, 4])


@pytest.mark.parametrize("name,many,opts", CASES)
def test_resident_equals_streamed(name, many, opts):
    from paper_2408_04066_gb300 import mfem
    cfg = config(name)
    xf = np.asarray(cfg["xfs"])
    opts = dict(dict(tile_rows=128, spmv_split=1, newton_max=6), **opts)
    ctx = mfem.Context.from_config(cfg, max_batch=many, **opts)
    alone = [ctx.solve_batch(xf[i:i + 1]) for i in range(len(xf))]
    p = ctx.profile()
    assert p["kernel_launches"] < p["pcg_launches"]          # one launch a solve
    out, stats = ctx.solve_batch(np.concatenate([xf] * (many // len(xf))))
    p = ctx.profile()
    assert p["kernel_launches"] > p["pcg_launches"]          # launches per iteration
    for b in range(len(out)):
        x, st = alone[b % len(xf)]
        assert np.array_equal(out[b], x[0])
        assert stats[b]["pcg_iters"] == st[0]["pcg_iters"] and stats[b]["newton_iters"] == st[0]["newton_iters"]
    ctx.close()


def test_iteration_cap():
    """A solve cut off by cg_max stops after exactly that many iterations a Newton step."""
    from paper_2408_04066_gb300 import mfem
    cfg = config("fig3000")
    ctx = mfem.Context.from_config(cfg, spmv_split=1, tile_rows=64, cg_max=3, newton_max=2, newton_tol=0.0, cg_tol=0.0)
    _, st = ctx.solve_batch(np.asarray(cfg["xfs"])[:1])
    assert st[0]["newton_iters"] == 2 and st[0]["pcg_iters"] == 6
    ctx.close()


@pytest.mark.parametrize("cap", [8192, 8193, 2**31 - 1])
def test_large_iteration_caps(cap):
    """Caps at and past the most iterations of one launch give the default cap's solve."""
    from paper_2408_04066_gb300 import mfem
    cfg = config("bar")
    res = []
    for opts in (dict(), dict(cg_max=cap)):
        ctx = mfem.Context.from_config(cfg, spmv_split=1, tile_rows=128, **opts)
        x, st = ctx.solve_batch(np.asarray(cfg["xfs"])[:1])
        res.append((x, st[0]["pcg_iters"], st[0]["newton_iters"], st[0]["converged"]))
        ctx.close()
    assert np.array_equal(res[0][0], res[1][0]) and res[0][1:] == res[1][1:] and res[0][3]


@pytest.mark.parametrize("saved", [False, True])
def test_64_row_blocks_without_a_search_of_them(saved, tmp_path, monkeypatch):
    """The shape search leaves 64-row blocks out, but the option and an earlier pick saved
    in the cache file still give them."""
    from paper_2408_04066_gb300 import mfem
    cfg = config("bar")
    xf = np.concatenate([np.asarray(cfg["xfs"])] * 160)[:160]
    f = tmp_path / "picks"
    if saved:
        monkeypatch.setenv("MFEM_AUTOTUNE_CACHE", str(f))
        ctx = mfem.Context.from_config(cfg, max_batch=160)
        ctx.solve_batch(xf)
        ctx.close()
        f.write_text(" ".join(f.read_text().split()[:-2] + ["64", "1"]) + "\n")
    ctx = mfem.Context.from_config(cfg, max_batch=160, tile_rows=0 if saved else 64)
    _, stats = ctx.solve_batch(xf)
    assert ctx.profile()["tile_rows"] == 64 and all(s["converged"] for s in stats)
    ctx.close()


@pytest.mark.parametrize("precond", ["two_level", "block_jacobi"])
def test_served_requests_that_join_a_resident_solve(precond):
    """A request alone in the server runs in the resident kernel a chunk at a time; requests
    that arrive while it runs make the table too large, and its solve goes on in the streamed
    kernels.  Every result still equals the same pose solved alone, bit for bit."""
    import time

    from paper_2408_04066_gb300 import mfem
    cfg = figure_config(50000, model="corot", seeds=range(16))
    xf = np.asarray(cfg["xfs"])
    opts = dict(tile_rows=256, spmv_split=1, precond=precond, max_batch=16)
    ctx = mfem.Context.from_config(cfg, **opts)
    alone = [ctx.solve_batch(x[None])[0][0] for x in xf]
    ctx.close()
    srv = mfem.Server(max_slots=16)
    mid = srv.add(mfem.Context.from_config(cfg, **opts))
    srv.wait(srv.submit(mid, xf[0]))                          # first launches, slot pools
    for pause_us in (300, 600, 1000, 1500, 2000, 3000):
        tickets = [srv.submit(mid, xf[0])]
        t = time.perf_counter()
        while (time.perf_counter() - t) * 1e6 < pause_us:
            pass
        tickets += [srv.submit(mid, x) for x in xf[1:]]
        for b, ticket in enumerate(tickets):
            out, _, _ = srv.wait(ticket)
            assert np.array_equal(out, alone[b]), (pause_us, b)
    srv.close()

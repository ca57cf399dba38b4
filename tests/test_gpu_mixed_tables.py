"""Several meshes in one call of which the first fits the chip and another does not:
the SpMV's shape is then searched on a group that is not the call's first, with more
poses than the first context has slots for."""
import numpy as np
import pytest

from synth import figure_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lead,other", [("mixed", "mixed"), ("mixed", "fp64"), ("fp64", "mixed")])
def test_shape_search_on_a_later_group(lead, other):
    from paper_2408_04066_gb300 import mfem
    cfgs = [dict(figure_config(3000, seeds=[5]), model="snh"),
            dict(figure_config(60000, seeds=range(12)), model="corot")]
    opts = dict(spmv_split=1)
    # one slot in the first context, twelve poses in the second: 12 x 26 blocks of 512 rows, past 152 SMs
    ctxs = [mfem.Context.from_config(c, precision=p, max_batch=len(c["xfs"]), **opts)
            for c, p in zip(cfgs, (lead, other))]
    outs, stats = mfem.solve_multi(ctxs, [c["xfs"] for c in cfgs])
    assert ctxs[0].profile()["tile_rows"] in (128, 256)
    again, stats2 = mfem.solve_multi(ctxs, [c["xfs"] for c in cfgs])
    for i, (cfg, p) in enumerate(zip(cfgs, (lead, other))):
        alone = mfem.Context.from_config(cfg, precision=p, max_batch=1, **opts)
        for b in range(len(cfg["xfs"])):
            x, st = alone.solve_batch(cfg["xfs"][b:b + 1])
            assert st[0]["converged"] and stats[i][b]["converged"]
            for k in ("newton_iters", "pcg_iters"):
                assert stats2[i][b][k] == st[0][k], (i, b, k)
            assert np.array_equal(again[i][b], x[0]), (i, b)
            assert np.array_equal(outs[i][b], x[0]), (i, b)
        alone.close()
    for c in ctxs:
        c.close()


def test_second_context_grows_between_calls():
    """The captured launches of a call hold the buffers of all its contexts: when the second
    one's slots are allocated anew, the next call of the same sizes uses the new ones."""
    from paper_2408_04066_gb300 import mfem
    cfgs = [dict(figure_config(20000, seeds=range(4)), model="corot"),
            dict(figure_config(60000, seeds=range(6)), model="corot")]
    ctxs = [mfem.Context.from_config(c, max_batch=len(c["xfs"]), tile_rows=128, spmv_split=1) for c in cfgs]
    xfs = [c["xfs"] for c in cfgs]
    first = [mfem.solve_multi(ctxs, xfs) for _ in range(3)]   # chunks of the default and the predicted lengths
    ctxs[1].solve_batch(np.concatenate([cfgs[1]["xfs"]] * 3))
    then = [mfem.solve_multi(ctxs, xfs) for _ in range(3)]
    for outs, stats in first[1:] + then:
        for i in range(2):
            assert np.array_equal(outs[i], first[0][0][i])
            assert [s["pcg_iters"] for s in stats[i]] == [s["pcg_iters"] for s in first[0][1][i]]
    for c in ctxs:
        c.close()


def test_search_when_only_the_whole_table_is_too_large(tmp_path, monkeypatch):
    """Meshes that fit the chip one by one but not together run in the streamed kernels: their
    shape is searched, on the larger group.  Together with a smaller one they fit: no search."""
    from paper_2408_04066_gb300 import mfem
    picks = tmp_path / "picks"
    monkeypatch.setenv("MFEM_AUTOTUNE_CACHE", str(picks))
    cfgs = [dict(figure_config(t, seeds=range(b)), model="corot") for t, b in ((3000, 1), (50000, 4), (60000, 5))]
    ctxs = [mfem.Context.from_config(c, max_batch=len(c["xfs"]), spmv_split=1) for c in cfgs]
    mfem.solve_multi(ctxs[:2], [c["xfs"] for c in cfgs[:2]])   # 1 x 2 + 4 x 22 blocks of 512 rows
    assert not picks.exists()
    outs, stats = mfem.solve_multi(ctxs[1:], [c["xfs"] for c in cfgs[1:]])   # 4 x 22 + 5 x 26, past 152 SMs
    lines = picks.read_text().splitlines()
    assert len(lines) == 1 and lines[0].split()[:2] == [str(ctxs[2].n), str(ctxs[2].m)]
    for i, cfg in enumerate(cfgs[1:]):
        alone = mfem.Context.from_config(cfg, max_batch=1, spmv_split=1, tile_rows=128)
        for b in range(len(cfg["xfs"])):
            assert np.array_equal(alone.solve_batch(cfg["xfs"][b:b + 1])[0][0], outs[i][b])
        alone.close()
    for c in ctxs:
        c.close()


def test_profile_of_two_precisions_in_one_call():
    """Resident solves of both precisions in one call are counted each by its own iterations and
    coarse bytes: the call's sums are those of the meshes solved alone."""
    from paper_2408_04066_gb300 import mfem
    cfgs = [dict(figure_config(3000, seeds=[5]), model="corot"), dict(figure_config(30000, seeds=[6]), model="corot")]
    ctxs = [mfem.Context.from_config(c, precision=p, max_batch=1, init="rigid")
            for c, p in zip(cfgs, ("fp64", "mixed"))]
    alone = []
    for c, cfg in zip(ctxs, cfgs):
        c.solve_batch(cfg["xfs"])
        alone.append(c.profile())
    mfem.solve_multi(ctxs, [c["xfs"] for c in cfgs])
    both = [c.profile() for c in ctxs]
    for k in ("pcg_launches", "coarse_launches", "pcg_iters", "pcg_bytes"):
        a, b = sum(p[k] for p in alone), sum(p[k] for p in both)
        assert abs(a - b) <= 1e-9 * a, k
    for c in ctxs:
        c.close()

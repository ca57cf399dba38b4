"""The bits of a pose do not depend on the calls before it or on the way it is solved,
with default options as well: a pose alone before and after a batch too large for the
chip (which times the SpMV's rows per block), in that batch, beside a mesh of the other
precision, and served."""
import numpy as np
import pytest

from synth import figure_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opts", [dict(precision="mixed"), dict(precision="fp64"), dict(precision="mixed", spmv_split=2),
                                  dict(precision="fp64", spmv_split=2)])
def test_same_bits_whatever_came_before(opts):
    from paper_2408_04066_gb300 import mfem
    cfg = dict(figure_config(50000, seeds=[3, 4]), model="snh")
    other = dict(figure_config(20000, seeds=[5]), model="corot")
    xf = np.asarray(cfg["xfs"])
    ctx = mfem.Context.from_config(cfg, max_batch=8, **opts)
    first = ctx.solve_batch(xf[:1])[0][0]
    batch, _ = ctx.solve_batch(np.concatenate([xf] * 4))      # 8 x 22 blocks of 512 rows: streamed
    p = ctx.profile()
    assert p["kernel_launches"] > p["pcg_launches"] and p["spmv_split"] == opts.get("spmv_split", 1)
    again = ctx.solve_batch(xf[:1])[0][0]
    lead = mfem.Context.from_config(other, max_batch=1, **dict(opts, precision="fp64" if opts["precision"] == "mixed" else "mixed"))
    beside = mfem.solve_multi([lead, ctx], [other["xfs"], xf[:1]])[0][1][0]
    for x in (batch[0], batch[6], again, beside):
        assert np.array_equal(x, first)
    srv = mfem.Server(max_slots=2)
    mid = srv.add(ctx)
    assert np.array_equal(srv.wait(srv.submit(mid, xf[0]))[0], first)
    srv.close()
    lead.close()

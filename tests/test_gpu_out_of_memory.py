"""A batch larger than the device holds is refused; its context holds no slots then, says so
where a state is read, and solves as before once a pose is set."""
import ctypes as C

import numpy as np
import pytest

from synth import bar_twist_config

pytestmark = pytest.mark.gpu


def test_refused_batch_leaves_a_usable_context():
    from paper_2408_04066_gb300 import mfem
    cfg = bar_twist_config()
    xf = np.asarray(cfg["xfs"])[:1]
    ctx = mfem.Context.from_config(cfg, precision="mixed", max_batch=1)
    ref = ctx.solve_batch(xf)[0][0]
    ctx.set_pose(xf[0])
    lib = mfem.load()
    out = np.empty((1, ctx.n, 3))
    # 2^31 - 1 poses: the poses' buffer alone is past the device memory, so the first allocation fails
    st = lib.mfem_solve_batch(ctx._ctx, C.c_void_p(xf.ctypes.data), 2**31 - 1, C.c_void_p(out.ctypes.data), 0, None)
    assert st == mfem.MFEM_ENOMEM
    for read in (ctx.get_elem, ctx.get_elem_static, ctx.get_state, ctx.solve):
        with pytest.raises(mfem.MfemError) as e:
            read()
        assert e.value.status == mfem.MFEM_EINVAL
    ctx.set_pose(xf[0])
    assert np.array_equal(ctx.solve()[0], ref)
    assert np.array_equal(ctx.solve_batch(np.concatenate([xf] * 2))[0][1], ref)
    assert ctx.get_elem()[0].shape == (ctx.m, 6)
    ctx.close()

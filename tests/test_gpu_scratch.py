"""Scratch that a context keeps between calls is given back before a call runs out of device memory."""
import numpy as np
import pytest

from dda_inputs import random_complex

pytestmark = pytest.mark.gpu

MB = 1 << 20


def test_kept_scratch_is_given_back_before_out_of_memory():
    """A near field leaves 0.5 GB of scratch behind.  With 150 MB free besides,
    a product of eight right-hand sides in double-float arithmetic, which takes
    over 250 MB, still runs, and so does the near field after it where there is
    room again; a product too large for both fails as before."""
    import torch
    import paper_1202_3424_gb300 as dda
    ctx = dda.Context(0)
    ctx.set_target(np.ones((48, 48, 48), np.uint8))
    ctx.set_materials([1.5 + 0.1j])
    ctx.prepare_size_parameter(1.0, dda.Precision.FP32_REFINED)
    n = ctx.info()["ndipoles"]
    R = 8
    k, e = np.tile([[0.6, 0.0, 0.8]], (R, 1)), np.tile([[0.0, 1.0, 0.0]], (R, 1)).astype(complex)
    x = torch.from_numpy(random_complex((R, 3, n), 3)).cuda()
    y, few = torch.empty_like(x), x[:1].clone()
    dda.dda_matvec_device(ctx.handle, 3, k[:1], e[:1], few, torch.empty_like(few))     # modules and small buffers
    P = random_complex((1, 3, n), 4)
    near = ctx.nearfield(1, k[:1], e[:1], P, [0.5] * 6)[1]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    filler = torch.empty(free - 150 * MB, dtype=torch.uint8, device="cuda")
    dda.dda_matvec_device(ctx.handle, 3, k, e, x, y)
    one = torch.empty_like(few)
    dda.dda_matvec_device(ctx.handle, 3, k[:1], e[:1], few, one)
    assert torch.equal(y[:1], one)
    with pytest.raises(dda.DdaError) as err:
        ctx.solve(1, np.tile(k[:1], (256, 1)), np.tile(e[:1], (256, 1)), want_P=False)
    assert err.value.status_name == "DDA_ERR_OOM"
    del filler
    torch.cuda.empty_cache()
    assert np.array_equal(ctx.nearfield(1, k[:1], e[:1], P, [0.5] * 6)[1], near)
    ctx.close()

"""One matrix alone against the same matrix many times over in one batch: the
root groups per warp, the FP64 tile size and the columns per gather or vector
warp follow the work of a height, and the bits must not.  Orders at the edges
of the lane-group sizes (4, 8, 16 and 32 lanes a root)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["uniform", "clustered"])
@pytest.mark.parametrize("n", [33, 64, 65, 129, 257, 600])
def test_height_width_does_not_change_bits(kind, n):
    from paper_2508_11467_gb300 import bdc, inputs
    copies = 96
    d, e = (torch.from_numpy(a).cuda() for a in inputs.make(kind, n, n))
    S, U, VT, info = bdc.svd(d, e, prec="fp64", leaf=16)
    plan = bdc.BatchPlan(d.repeat(copies), torch.cat([e, e.new_zeros(1)]).repeat(copies), [n] * copies, prec="fp64",
                         leaf=16)
    plan.launch()
    torch.cuda.synchronize()
    assert info == 0 and int(plan.info.abs().max()) == 0
    for one, many in ((S, plan.S), (U, plan.U), (VT, plan.VT)):
        many = many.reshape(copies, -1)
        flat = (one.t() if one.dim() == 2 and one.stride(0) == 1 else one).reshape(-1)
        assert bool((many == flat).all())
    plan.close()


@pytest.mark.parametrize("n", [33, 36, 37, 65, 130, 601])
def test_fp32_product_tiles_do_not_change_bits(n):
    """The FP32 products by 32 x 32 tiles (one matrix) and by the tiles of a
    full chip (many copies): every output sums its terms in the same order."""
    from paper_2508_11467_gb300 import bdc, inputs
    d, e = (torch.from_numpy(a).cuda() for a in inputs.make("uniform", n, n))
    e = torch.cat([e, e.new_zeros(1)])
    out = []
    for copies in (1, 200):
        plan = bdc.BatchPlan(d.repeat(copies), e.repeat(copies), [n] * copies, leaf=16, dtype=torch.float32)
        plan.launch()
        torch.cuda.synchronize()
        assert int(plan.info.abs().max()) == 0
        out.append([t.clone().reshape(copies, -1) for t in (plan.S, plan.U, plan.VT)])
        plan.close()
    for one, many in zip(*out):
        assert bool((many == one).all())

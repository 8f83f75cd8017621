"""grad_W + grad_X of sizes at the line between one launch and two, against the two single calls.

Another split of an fp32 sum changes it by about 1e-6 of the sum of magnitudes, which moves the bf16 result by at most one unit in
the last place (2^-7 of the value at the start of a binade) wherever it is not much smaller than those.
"""
import pytest

from paper_2409_09099_b200 import synth
from tests.gpu_util import dbf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("minimal", [False, True])
@pytest.mark.parametrize("O,I,T,fp8,dense_copy", [(2560, 1280, 640, False, True), (512, 7040, 1792, False, True),
                                                  (384, 8704, 128, False, False), (2176, 5376, 128, False, True),
                                                  (4096, 4352, 512, True, True), (3968, 896, 768, True, False),
                                                  (6016, 1152, 5504, False, True), (5248, 768, 8832, False, True)])
def test_gradients_at_the_line(O, I, T, fp8, dense_copy, minimal):
    from paper_2409_09099_b200 import binding as B
    from paper_2409_09099_b200.layer import SsteLinear
    ctx = B.Context(0, minimal_workspace=minimal)
    try:
        W = dbf16(synth.gaussian_bf16(O + 61, (O, I), 0.02))
        X = dbf16(synth.gaussian_bf16(O + 62, (T, I), 1.0))
        dY = dbf16(synth.gaussian_bf16(O + 63, (T, O), 1e-2))
        lin = SsteLinear(ctx, W, T, tensor_id=4, seed=17, fp8=fp8, dense_copy=dense_copy)
        lin.init_beta(); lin.prune(); lin.forward(X)
        for rep in range(2):                                 # the tickets of split tiles must be left at zero
            lin.dX.fill_(7.0); lin.dW.fill_(7.0)
            before = B.launch_count()
            dX, dW = (t.clone() for t in lin.backward(dY, step=3))
            launched = B.launch_count() - before
            ref_w, ref_x = lin.grad_weight().float(), lin.grad_input(dY).float()
            for got, ref in ((dW.float(), ref_w), (dX.float(), ref_x)):
                assert bool(((got - ref).abs() <= 2.0 ** -7 * ref.abs() + 1e-5 * ref.abs().max()).all())
        # the two largest sizes take two launches; so does a weight that the minimal workspace has no room to expand
        one = O < 5000 and (dense_copy or not minimal)
        assert ctx.lib.sste_layer_grads_joint(ctx.handle, lin._desc.at) == one
        in_front = 2 if fp8 else 1                           # (max|dY| and) the sparsification of dY
        expanded = not dense_copy and not minimal
        assert launched == in_front + expanded + (1 if one else 2)
        assert ctx.poll_device_status() == 0
    finally:
        ctx.close()

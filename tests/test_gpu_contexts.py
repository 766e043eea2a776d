"""Several contexts in one process: a kernel's shared-memory limit belongs to the device, so a context of shorter windows
must not lower it for one of longer windows that was created before."""
import dataclasses

import pytest

torch = pytest.importorskip("torch")

from paper_2403_18661_gb300 import abi, inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("net", [inputs.TINY_NET, inputs.RESNET34_NET])
@pytest.mark.parametrize("precision", [abi.AFG_BF16, abi.AFG_FP32])
def test_a_context_of_shorter_windows_leaves_the_others_alone(net, precision):
    w = inputs.make_weights(net, 3)
    y = torch.randn((2, 8192), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    ctx = {n: abi.Context(dataclasses.replace(inputs.PLAIN_64S, net=net, win_len=n), w, precision=precision)
           for n in (3072, 1024)}
    for n in (3072, 1024):
        z = ctx[n].infer_windows(y, 0, 128, 9)
        ctx[n].sync()
        alone = abi.Context(dataclasses.replace(inputs.PLAIN_64S, net=net, win_len=n), w, precision=precision)
        assert torch.equal(alone.infer_windows(y, 0, 128, 9), z)
        alone.sync()
        alone.close()
    for c in ctx.values():
        c.close()

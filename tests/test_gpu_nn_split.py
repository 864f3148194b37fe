"""Whole gradients of the network at sizes where the backward pass changes route:
the decoder's d(cat) split by the GEMM's epilogue (tcgen05 kernels, 32-channel
levels and above) or by a separate pass (16- and 48-channel levels), eight-
channel pooling kernels, ragged patch tiles, split-k reductions of four
columns.  Against the float64 oracle with its bfloat16 operand rounding, at the
tolerances of the other whole-network gradients (1e-2 of the gradient's norm, 0.1
per tensor: the effect of flipped bfloat16 roundings)."""
import numpy as np
import pytest

import oracle.nn as onn
from gpu_helpers import rel_l2, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base,levels,n,h,w", [(16, 2, 2, 24, 40), (32, 1, 3, 18, 22), (32, 3, 1, 40, 72),
                                               (48, 2, 2, 12, 20), (64, 2, 1, 36, 28)])
def test_gradient_at_route_edges(base, levels, n, h, w):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_17518_gb300 import build
    from paper_2403_17518_gb300.ops import Context

    build()
    spec = onn.UNetSpec(base, levels)
    rng = np.random.Generator(np.random.PCG64(3))
    x = rng.standard_normal((n, h, w)).astype(np.float32)
    y = rng.standard_normal((n, h, w)).astype(np.float32)
    ctx = Context(h, w, 10.0, 1e-3, 4)
    ctx.net_init(base, levels, 11)
    loss, grad = ctx.deblur_grad(to_dev(x), to_dev(y))
    grad = to_host(grad)
    ctx.close()
    flat = onn.init_params(spec, 11)
    out, cache = onn.forward(flat, x[:, None].astype(np.float64), spec)
    ref_loss, dout = onn.mse(out, y[:, None].astype(np.float64))
    ref = onn.backward(flat, cache, dout, spec)
    assert abs(loss - ref_loss) <= 1e-3 * ref_loss
    assert rel_l2(grad, ref) <= 1e-2
    k = 0
    for name, kind, ci, co in onn.param_specs(spec):
        cnt = int(np.prod(onn.weight_shape(kind, ci, co))) + co
        assert rel_l2(grad[k:k + cnt], ref[k:k + cnt]) <= 0.1, name
        k += cnt

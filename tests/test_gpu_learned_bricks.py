"""Gradients of the correction network where the weight-gradient kernel's
bricks of 16 x 4 x 4 voxels are ragged: extents below, at and beyond a brick
at every level (the bottom level has a quarter of them), against the float64
reference with the kernels' bfloat16 storage rounding.  Tolerance: float32
against float64 accumulation of products of bfloat16 values (a few 1e-7) and
rare rounding-boundary flips of the bfloat16 storage (2^-8 each), the 1e-2
per layer of the 8^3 test."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import unet as ou
from paper_1901_07892_gb300 import wsi
from test_gpu_learned import NAMES, _bf16, _built, _pack_grads, _unpack  # noqa: F401


@pytest.mark.parametrize("shape", [(4, 4, 4), (4, 12, 20), (12, 8, 36), (20, 4, 64)])
def test_gradients_on_ragged_bricks(shape):
    c0, c1, c2 = 16, 32, 64
    net = wsi.UNet(*shape, c0, c1, c2, seed=5)
    rng = np.random.default_rng(1)
    p = _bf16(net.params())
    net.set_params(p)
    x = _bf16(rng.standard_normal(shape + (3,)).astype(np.float32))
    t = rng.standard_normal(shape).astype(np.float32)
    net.forward(x)
    loss = net.backward(t)
    g = net.grads()
    P = _unpack(p, c0, c1, c2)
    ref, tape = ou.forward(P, np.transpose(x, (3, 0, 1, 2)).astype(np.float64), rnd=ou.bf16)
    assert loss == pytest.approx(ou.loss(ref, t[None].astype(np.float64)), rel=2e-3)
    gr, _ = ou.backward(P, tape, ref, t[None].astype(np.float64), rnd=ou.bf16)
    G = _pack_grads(gr, c0, c1, c2)
    off, shapes, errs = 0, ou.layer_shapes(3, c0, c1, c2), {}
    for name in NAMES:
        co, ci = shapes[name]
        n = 27 * co * (16 if name == "a1" else ci) + co
        a, b = g[off:off + n], G[off:off + n]
        errs[name] = float(np.linalg.norm(a - b) / np.linalg.norm(b))
        off += n
    errs["head"] = float(np.linalg.norm(g[off:] - G[off:]) / np.linalg.norm(G[off:]))
    print(shape, errs)
    assert max(errs.values()) < 1e-2, errs
    net.close()

"""GPU test of the tcgen05 convolution at the edges of its tiles (8 x 16 voxels
by 1 to 8 planes, input channel blocks of 16, output channel blocks of 16 to
64): forward pass and gradients on extents around them, against the mma.sync
implicit GEMMs on the same network (every layer's convolution and data
gradient there has another kernel, tiling and summation order)."""
import numpy as np
import pytest

from paper_2412_16843_gb300 import cdi, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2412_16843_gb300 import build
    build.build()
    cdi.load()


@pytest.mark.parametrize("n", [(8, 8, 8), (72, 16, 8), (16, 136, 24), (40, 24, 72), (128, 112, 8)],
                         ids=lambda n: "x".join(map(str, n)))
def test_convolution_tiles_match_the_mma_kernels(n):
    """Both sum the same BF16 products in FP32 and round each layer to BF16
    once, so they differ where a sum rounds the other way: a BF16 step is
    2^-8, a rounding flips in well under 1 % of the voxels, and the output
    differs by less than 2^-8 sqrt(0.01) = 4e-4 a layer: 2e-3 over the seven
    (relative, L2).  A voxel taken from the wrong place moves it by O(1)."""
    rng = np.random.default_rng(sum(n))
    shape = (n[2], n[1], n[0])
    x, t = rng.standard_normal(shape + (2,)), rng.standard_normal(shape)
    out = []
    for kernel in (1, 0):
        net = cdi.Unet(n)
        net.set_conv_kernel(kernel)
        net.set_params(inputs.unet_initial_params(3))
        y = net.forward(x)
        out.append((y, net.train_step(x, t, want_grads=True)[1]))
    for k, tol in ((0, 2e-3), (1, 2e-2)):  # gradients: ReLU masks flip too, within the bar of the gradient parity
        a, b = out[0][k], out[1][k]
        assert np.linalg.norm(a - b) <= tol * np.linalg.norm(b)

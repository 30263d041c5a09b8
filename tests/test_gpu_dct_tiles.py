"""The DCT preconditioner's products in each of their three builds, at ragged masked sizes, pixel
by pixel: 64-wide tiles with eight stages (at most half as many 128-wide tiles as SMs), 128-wide
tiles with six stages (at most as many tiles as SMs) and with three, two blocks to an SM (more).

Reference: the same transform as plain FP64 matrix products.  Bar: every operand (r, the cosine
matrices, the intermediate planes) is the sum of two BF16 numbers, good to 2^-17 of its size, and
such roundings are white noise.  What enters before the division by the Laplacian's eigenvalues L
is seen through 1 / L, what enters after it is not, so with four operands on either side
||got - s|| < 4 * 2^-17 (||r|| rms(1 / L) + ||s||); a CPU emulation of the splits reaches 0.06 to
0.33 of that at 130 x 65 to 1100 x 900.  The noise is spread over the map: a pixel may be eight
times its r.m.s. value off."""
import math

import numpy as np
import pytest
import torch

from paper_2203_13675_gb300 import native, synth

pytestmark = pytest.mark.gpu


def _dct(n):
    k = torch.arange(n, dtype=torch.float64, device="cuda")[:, None]
    x = torch.arange(n, dtype=torch.float64, device="cuda")[None, :]
    c = torch.cos(math.pi * k * (x + 0.5) / n) * math.sqrt(2.0 / n)
    c[0] = math.sqrt(1.0 / n)
    return c


@pytest.mark.parametrize("H,W,build", [(130, 65, "64"), (700, 333, "64"), (1100, 900, "64"), (1190, 1153, "128, six"),
                                       (700, 2000, "128, six"), (1300, 1900, "128, three"), (2049, 1111, "128, three")])
def test_apply_on_every_tile_shape(H, W, build):
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    tiles = -(-H // 128) * -(-W // 128)
    assert build == ("64" if 2 * tiles <= nsm else "128, six" if tiles <= nsm else "128, three")
    m = synth.phase_map(H, W, 7 + W, noise=0.6, mask_frac=0.05)
    psi, mask = torch.from_numpy(np.ascontiguousarray(m.psi)).cuda(), torch.from_numpy(m.mask).to(torch.uint8).cuda()
    dx, dy = native.ulp_wrapped_diffs(psi)
    U, V, b = native.ulp_weights(torch.zeros_like(psi), dx, dy, mask, p=1.0, eps=1e-2)
    got = native.ulp_precond_apply("dct", U, V, b, mask=mask)
    ch, cw = _dct(H), _dct(W)
    lam = (2 - 2 * torch.cos(math.pi * torch.arange(H, dtype=torch.float64, device="cuda") / H))[:, None] + \
        (2 - 2 * torch.cos(math.pi * torch.arange(W, dtype=torch.float64, device="cuda") / W))[None, :]
    lam[0, 0] = math.inf
    full = ch.T @ ((ch @ b @ cw.T) / lam) @ cw
    ref = torch.where(mask != 0, 0.0, full)
    bar = 4 * 2.0 ** -17 * float(torch.linalg.norm(b) * (1 / lam).square().mean().sqrt() + torch.linalg.norm(full))
    assert float(torch.linalg.norm(got - ref)) < bar
    assert float((got - ref).abs().max()) < 8 * bar / math.sqrt(H * W)
    assert bool((got[mask != 0] == 0).all())

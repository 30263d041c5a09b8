"""The wavefront sweeps at the edges of their shared-memory rings: widths around one
8-column chunk and one 64-column ring, bands of one, 31, 32 and 33 rows, and more
32-row bands than the chip holds at once, against the oracle's sequential sweeps.

Tolerance: each value is the oracle's arithmetic up to the rounding of the precomputed
coefficients, 1e-12 of the largest value, as for the other sweep tests."""
import numpy as np
import pytest
import torch

import oracle
from paper_2203_13675_gb300 import native, synth

pytestmark = pytest.mark.gpu
KINDS = {"ilu0": oracle.M_ILU0, "ssor": oracle.M_SSOR}


@pytest.mark.parametrize("kind", ["ilu0", "ssor"])
@pytest.mark.parametrize("H,W", [(3, 7), (31, 8), (32, 9), (33, 2), (65, 63), (70, 64), (34, 65), (129, 73),
                                 (40, 200), (20011, 11)])
def test_apply_at_ring_edges(kind, H, W):
    m = synth.phase_map(H, W, 3 + H + W, noise=0.7, mask_frac=0.05 if min(H, W) > 30 else 0.0, ramp=0.1)
    dx, dy = oracle.wrapped_diffs(m.psi)
    U, V = oracle.weights(np.zeros((H, W)), dx, dy, m.mask, 1.0, 0.01)
    r = np.random.default_rng(W).normal(size=(H, W))
    ref = oracle.precond_apply(KINDS[kind], oracle.assemble(U, V, dx, dy), r, omega=1.0)
    dev = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (U, V, r)]
    got = native.ulp_precond_apply(kind, *dev).cpu().numpy()
    np.testing.assert_allclose(got, ref, rtol=1e-12, atol=1e-12 * np.abs(ref).max())

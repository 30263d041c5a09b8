"""The FP64 flexible CG with more tiles than a block of its phase B adds up by itself
(small tile_rows, or very large maps), where small kernels add the tile partials first: one tile
below the line, one above it, a ragged last round of partials, and several rounds.

Reference: the same call on the plan's own tiles, whose sums are grouped by other tiles.  After
12 iterations red-black SSOR differs by the rounding of its scalars (bar 1e-10 of the largest
value); multigrid works in 32 bits inside, where a last bit may round otherwise (bar 1e-5).  A
single missing or doubled partial of n is a change of about 1 / n.  (DCT adds its sums by the
kernels of red-black SSOR; its products' 16-bit operands leave a constant offset free, for which
no bar is known.)"""
import numpy as np
import pytest
import torch

from paper_2203_13675_gb300 import native, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,bar", [("rbssor", 1e-10), ("mg", 1e-5)])
@pytest.mark.parametrize("H,W,rows", [(4096, 64, 1), (4097, 64, 1), (2500, 130, 1), (6001, 200, 1), (700, 2000, 2)])
def test_sums_of_many_tiles(H, W, rows, kind, bar):
    psi = torch.from_numpy(np.ascontiguousarray(synth.phase_map(H, W, 40 + W, noise=0.5).psi)).cuda()
    got = []
    for opt in (dict(tile_rows=rows), dict(tile_rows=rows, profile=2), dict()):
        plan = native.Plan(H, W, outer_tol=0.0, **opt)
        phi, st = plan.unwrap(psi, None, p=1.0, precond=kind, tol=1e-14, max_outer=1, max_inner=12)
        got.append((phi, st["inner"], st["status"]))
    (a, ia, sa), (h, ih, sh), (b, ib, sb) = got
    assert ia == ib == [12] and sa == sb == native.ULP_WARN_MAXITER
    assert (ih, sh) == (ia, sa) and torch.equal(h, a)  # host-driven: the same kernels
    assert float((a - b).abs().max()) < bar * float(b.abs().max())

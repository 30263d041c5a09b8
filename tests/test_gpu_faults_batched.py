"""A bounded wait that runs out in a batch whose blocks hold tiles of several maps: every thread
of a block must leave together, whichever map's wait it was.  As in test_gpu_faults.py a bound
of one nanosecond makes the first wait give up; the call returns ULP_ERR_TIMEOUT, and the next
call in the same context runs normally."""
import numpy as np
import pytest
import torch

from paper_2203_13675_gb300 import native, synth

pytestmark = pytest.mark.gpu

SIZES = [(64, 64), (37, 53), (130, 67), (96, 128), (18, 40), (64, 200), (33, 65), (50, 20)] * 3


@pytest.mark.parametrize("rows", [0, 16])  # on the chip; streaming, eight tiles of several maps to a block
@pytest.mark.parametrize("mixed", [0, 1])
def test_bounded_wait_runs_out_in_a_batch(mixed, rows):
    maps = []
    for k, (h, w) in enumerate(SIZES):
        psi = torch.from_numpy(np.ascontiguousarray(synth.phase_map(h, w, 300 + k, noise=0.4).psi)).cuda()
        maps.append({"psi": psi, "mask": None, "phi": torch.empty_like(psi), "p": 1.0, "eps": 1e-2})
    kw = dict(sizes=SIZES, outer_tol=0.0, precision=mixed, tile_rows=rows)
    for _ in range(3):
        plan = native.Plan(None, spin_timeout_s=1e-9, **kw)
        with pytest.raises(native.UlpError) as ei:
            plan.unwrap_batched(maps, precond="jacobi", tol=1e-6, max_outer=2)
        assert ei.value.status == native.ULP_ERR_TIMEOUT, ei.value
        plan.close()
        plan = native.Plan(None, **kw)
        rc, stats = plan.unwrap_batched(maps, precond="jacobi", tol=1e-6, max_outer=2)
        assert rc == 0 and all(s["status"] == native.ULP_OK and s["outer"] == 2 for s in stats)
        plan.close()

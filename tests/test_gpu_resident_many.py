"""The resident Jacobi / identity solvers with three and more maps in a block: the maps stop
at different iterations and, in FP64, recompute their true residual at different ones, so a
block adds up sums of some of its maps and not of others.  Every map against its own solve on
a plan whose 16-row tiles stream their planes (the bars of the other tests of these solvers:
counts within 2, at relative residual 1e-6 a difference below 1e-4 rad RMS), and the whole
batch again, which must give the same bits."""
import numpy as np
import pytest
import torch

from paper_2203_13675_gb300 import native, synth

pytestmark = pytest.mark.gpu


def _sizes(which):
    if which == "one large, twelve strips":  # nine tiles of four rows to a block, three to a strip
        return [(480, 640)] + [(12, 60)] * 12
    rng = np.random.default_rng(4)
    return [(int(h), int(w)) for h, w in zip(rng.integers(4, 15, 256), rng.integers(5, 61, 256))]


# (M = I on maps of a few dozen pixels runs past as many iterations as there are unknowns, where
# rounding decides its count: no bar is known for it, and it takes the first batch only)
@pytest.mark.parametrize("kind,which", [("jacobi", "one large, twelve strips"), ("jacobi", "256 small"),
                                        ("identity", "one large, twelve strips")])
@pytest.mark.parametrize("mixed", [0, 1])
def test_many_maps_to_a_block(kind, mixed, which):
    sizes = _sizes(which)
    tiles = [-(-h // 4) * -(-w // 64) for h, w in sizes]
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    per = -(-sum(tiles) // nsm)
    ends = np.cumsum(tiles)
    first = np.searchsorted(ends, np.arange(0, ends[-1], per), side="right")
    last = np.searchsorted(ends, np.minimum(np.arange(0, ends[-1], per) + per, ends[-1]) - 1, side="right")
    assert (last - first + 1).max() >= 3  # what the test is about
    maps = []
    for k, (h, w) in enumerate(sizes):
        m = synth.phase_map(h, w, 900 + k, noise=0.2 + 0.6 * (k % 7) / 6)
        psi = torch.from_numpy(np.ascontiguousarray(m.psi)).cuda()
        maps.append({"psi": psi, "mask": None, "phi": torch.empty_like(psi), "p": float(k % 2), "eps": 1e-2})
    plan = native.Plan(None, sizes=sizes, outer_tol=0.0, precision=mixed)
    _, stats = plan.unwrap_batched(maps, precond=kind, tol=1e-6, max_outer=2)
    once = [d["phi"].clone() for d in maps]
    _, again = plan.unwrap_batched(maps, precond=kind, tol=1e-6, max_outer=2)
    assert [s["inner"] for s in again] == [s["inner"] for s in stats]
    assert all(torch.equal(a, d["phi"]) for a, d in zip(once, maps))
    one = {}
    for (h, w), d, st in zip(sizes, maps, stats):
        if (h, w) not in one:
            one[h, w] = native.Plan(h, w, outer_tol=0.0, precision=mixed, tile_rows=16)
        ref, rst = one[h, w].unwrap(d["psi"], None, p=d["p"], precond=kind, tol=1e-6, max_outer=2)
        assert st["status"] == rst["status"]
        for a, b in zip(st["inner"], rst["inner"]):
            assert abs(a - b) <= (2 if kind == "jacobi" else max(2, int(0.05 * b))), ((h, w), st["inner"], rst["inner"])
        e = d["phi"] - ref
        assert float(((e - e.mean()) ** 2).mean().sqrt()) < 1e-4

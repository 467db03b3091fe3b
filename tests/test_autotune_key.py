"""The tuner's cache key on the CPU: grids that differ in the number of sims or levels (which
decide what forms fit) have entries of their own, and an entry written for other kernels
(the key without the revision, as caches of the earlier kernels have it) is not applied."""
import json

from test_autotune_cache import FakeGrid, table

from paper_1808_04099_gb300 import autotune


def tune(path, best, n_sims=1, max_level=0):
    g = FakeGrid(table(best))
    g.spec.n_sims, g.spec.max_level = n_sims, max_level
    autotune.tune(g, iters=3, cache_path=path, device_name="d")
    return g


def test_sims_and_levels_have_entries_of_their_own(tmp_path):
    path = str(tmp_path / "c.json")
    assert tune(path, (3, 1, 1)).shape == (3, 1, 1)
    for sims, levels, best in ((8, 0, (1, 2, 1)), (1, 1, (2, 1, 1)), (8, 1, (0, 1, 1))):
        g = tune(path, best, sims, levels)
        assert g.solves > 0 and g.shape == best
    assert len(json.load(open(path))) == 4
    assert tune(path, (0, 2, 2), 8, 0).solves == 0  # from its entry


def test_entries_of_earlier_kernels_are_not_applied(tmp_path):
    path = tmp_path / "c.json"
    shapes = ";".join(f"{a},{b},{c}" for a, b, c in autotune.SHAPES)
    old = {f"d|B16|prec1|cubes1024|shapes{shapes}": {"best": [2, 4, 1], "times": {"2,4,1": 1.0}}}
    path.write_text(json.dumps(old))
    g = tune(str(path), (3, 1, 1))
    assert g.solves > 0 and g.shape == (3, 1, 1)

"""bench.py names the search kernel that the handle ran, not the one its phase
usually holds.  CPU only."""
import importlib.util
import os
import types

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("search,phase,tests,kernel", [
    (0, "search", None, "search_kernel"), (1, "search", None, "filter_search_kernel"),
    (1, "search", 12.0, "filter_search_kernel"), (2, "search", None, "pairs_search_kernel"),
    (3, "tile", None, "tile_search_kernel"), (4, "tile", 100.0, "tile_pruned_kernel"),
    (2, "move", None, "move_kernel"),
])
def test_kernel_of_the_dominant_phase(search, phase, tests, kernel):
    spec = importlib.util.spec_from_file_location("kmc_bench", os.path.join(ROOT, "bench.py"))
    bench = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(bench)
    phases = {p: 1.0 for p in bench.PHASE_NAMES}
    phases[phase] = 10.0
    r = dict(prof=phases, pairs=1e5, cand=100.0, tile_tests=tests, search=search,
             info=types.SimpleNamespace(n_search_cells=1000, n_bins=100))
    roof, _ = bench.roofline_of(dict(n=1_000_000, precision=32), r, 1, 152, {}, "test", "none")
    assert roof["kernel"] == kernel

"""The largest caches a handle accepts: B + M candidates of a layer in the shared memory of one selection cluster."""
import pytest

from paper_2603_05959_b200 import binding as B

from test_abi import _cfg, lib  # noqa: F401  (the fixture builds the library)


# (grid, aux tokens, candidates that have to be accepted): frames of one token to frames that fill a third of the cache
@pytest.mark.parametrize("grid,n_special,candidates", [((1, 1), 0, 83104), ((8, 8), 5, 82912), ((10, 10), 27, 82752), ((13, 11), 5, 82656),
                                                       ((23, 31), 5, 80768), ((28, 37), 5, 79728), ((37, 37), 5, 78624),
                                                       ((45, 44), 20, 76608), ((64, 64), 5, 69712), ((64, 128), 5, 56320),
                                                       ((120, 120), 5, 35984), ((1, 1), 9000, 70016)])
def test_candidates_accepted(lib, grid, n_special, candidates):  # noqa: F811
    M = n_special + grid[0] * grid[1]
    need = lambda n: lib.ovggt_workspace_bytes(_cfg(n_heads=1, n_special=n_special, grid_h=grid[0], grid_w=grid[1], budget=n - M,
                                                    anchor_tokens=0, dtype=B.DTYPE_BF16))
    assert need(candidates) > 0
    assert need(candidates + 1000) == 0                  # (and beyond it a handle is refused, not the first step)


def test_camera_candidates_accepted(lib):  # noqa: F811
    cfg = lambda b: _cfg(n_heads=1, camera_head=1, n_special=1, grid_h=0, grid_w=0, anchor_tokens=0, budget=b)
    assert lib.ovggt_workspace_bytes(cfg(83120 - 1)) > 0

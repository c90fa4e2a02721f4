"""GPU parity of the clip backward at chunk sizes round its 128-row tiles and their 64-row halves: the query columns
of the dk/dv blocks that are not live, key rows a group does not see, one step and many."""
import pytest

from paper_2509_22622_b200 import synth

import test_gpu_bwd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("grid_h,grid_w,ctx,clip_chunks,window", [
    (1, 16, 0, 2, 2),       # a few rows
    (8, 8, 1, 3, 2),        # exactly a half
    (5, 13, 0, 1, 1),       # one row into the second half, one step
    (1, 127, 2, 2, 1),
    (8, 16, 1, 2, 2),       # exactly a tile
    (3, 43, 0, 3, 3),       # one row into the second tile
    (1, 193, 1, 2, 2),      # one row into its second half
])
def test_chunks_round_the_tiles(oracle_mod, D, grid_h, grid_w, ctx, clip_chunks, window):
    wl = synth.Workload("bwd_%dx%d" % (grid_h, grid_w), 1, 2, D, grid_h, grid_w, 1, 1, window + clip_chunks - 1, n_chunks=0,
                        seed=300 + grid_h * grid_w)
    test_gpu_bwd.test_clip_backward_matches_oracle(oracle_mod, wl, ctx, clip_chunks, window)

"""The executed products behind the bench line's roofline, counted for the tile
shapes that a circuit reports, as the bench counts them."""
import os
import sys

import pytest

from paper_1202_1350_gb300 import circuits, vc

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402

BY_SIZE = {"pr_chunk_log": vc.VC_TILE_BY_SIZE, "gn_chunk_log": vc.VC_TILE_BY_SIZE,
           "line_chunk_log": vc.VC_TILE_BY_SIZE, "eval_chunk_log": 11, "pr_split_log": vc.VC_SPLIT_WIDEST}


def test_f2_2e20():
    w, k = circuits.f2(20)
    assert bench.executed_work(w, k, BY_SIZE) == bench.executed_work(w, k) == 37_626_399


@pytest.mark.parametrize("general", [7, 12])
def test_the_general_chunk_does_not_count_for_the_line(general):
    w, k = circuits.f2(20)
    assert bench.executed_work(w, k, dict(BY_SIZE, gn_chunk_log=general)) == 37_626_399
    fixed = dict(BY_SIZE, gn_chunk_log=general, line_chunk_log=13)
    assert bench.executed_work(w, k, fixed) == 37_626_399


# coordinates a thread folds in registers: chunk - 7 where the chunk has more than 7
@pytest.mark.parametrize("n,widest,line,chunk", [(14, 14, None, 12), (12, 16, None, 13), (17, 17, None, 13),
                                                 (20, 22, None, 13), (21, 22, None, 14), (22, 22, None, 15),
                                                 (24, 24, None, 15), (22, 22, 13, 13), (14, 14, 13, 13), (20, 20, 9, 9)])
def test_line_chunks(n, widest, line, chunk):
    tiles = BY_SIZE if line is None else dict(BY_SIZE, line_chunk_log=line)
    assert bench.line_chunk_log(n, widest, tiles) == chunk

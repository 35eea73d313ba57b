"""The served run's roofline counts what a start has to move: every input once
and every output once, whatever the schedule's steps would."""
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import bench
from paper_2408_05962_gb300.serving import Request


def test_served_bytes():
    a = Request(kind="allreduce", P=8, hierarchy=[2, 4], bytes_per_rank=8 * 10 * 4 + 3, dtype="f32")
    b = Request(kind="allgather", P=16, hierarchy=[4, 4], bytes_per_rank=16 * 6 * 2, dtype="bf16")
    a.d, a.hbm_bytes = 10, 5000
    b.d, b.hbm_bytes = 6, 700
    # 8 ranks read and write 320 bytes each; 16 ranks read 12 bytes and write 192
    assert bench.served_bytes([a, b]) == (5700, 2 * 8 * 320 + 16 * 12 + 16 * 192)
    assert bench.served_bytes([]) == (0, 0)


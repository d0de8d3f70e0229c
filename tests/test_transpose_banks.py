"""The transpose of Cg reads columns of a shared tile, lane l the rows 2 l and 2 l + 1: with the
tile's row pitch no two lanes may meet in one of the 32 four-byte banks with different words."""
import os
import re

HOST = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2506_01260_gb300", "csrc", "sn_tc_host.cu")


def test_column_reads_fall_in_distinct_banks():
    pitch = int(re.search(r"__nv_bfloat16 tile\[64\]\[(\d+)\]", open(HOST).read()).group(1))
    assert pitch >= 128                                    # k <= 128 columns
    for half in (0, 1):
        for j in range(128):
            words = {2 * ((2 * lane + half) * pitch + j) // 4 for lane in range(32)}
            assert len({w % 32 for w in words}) == len(words)

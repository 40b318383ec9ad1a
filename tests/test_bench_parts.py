"""bench.py's label and bound of the tensor-core P2P follow the operand parts that the tree chose."""
import pytest

import bench


# sources and stages of 81920 panels (P 7, Ncrit 512) and of 1280 with ranges of a few sources
@pytest.mark.parametrize("sources,f16,tf32", [(4408095, 285067, 555479), (105060, 7399, 13546)])
def test_parts_from_the_stage_count(sources, f16, tf32):
    info = dict(p2p_group_sources=sources)
    assert bench.p2p_f16_parts(dict(info, p2p_stages=f16))
    assert not bench.p2p_f16_parts(dict(info, p2p_stages=tf32))

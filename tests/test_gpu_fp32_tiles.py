"""Which FP32 tiles are accepted: queries, two slabs with their ids and the
rows' buffers within 220 KB."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,C,k,most", [
    (32, 32, 200, 64), (64, 128, 10, 32), (64, 128, 200, 16), (128, 64, 10, 64), (128, 64, 60, 32),
    (128, 64, 200, 16), (96, 32, 200, 32), (20, 128, 200, 32), (100, 64, 60, 32), (160, 128, 10, 8),
    (256, 64, 10, 32), (256, 64, 60, 16), (256, 64, 200, 8),
])
def test_tiles_up_to_the_memory_limit(d, C, k, most):
    from paper_2601_11808_gb300.sivf import Index, SivfError
    ix = Index(d, 4, C, 1024, 64)
    for tq in (8, 16, 32, 64):
        tile = {"queries_per_tile": tq, "slabs_per_chunk": 4, "items_per_sm": 2, "select_slabs": 0,
                "nearest_first": 0}
        if tq > most:
            with pytest.raises(SivfError):
                ix.set_tile("fp32", 70, k, 3, tile)
            continue
        ix.set_tile("fp32", 70, k, 3, tile)
        assert ix.get_tile("fp32", 70, k, 3) == tile
    ix.close()

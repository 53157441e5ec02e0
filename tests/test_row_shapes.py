"""CPU model of the row tiles' copies (test_rowio_layout.py) and of the column
pass's lanes (test_colrs_layout.py) at the CTA shapes of tiling 0, its
defect-correction form's, and the two-column CTA at L = 2048: offsets equal
the index map, every access stays in the tile and in the spectrum, and no
bank conflicts."""
import pytest

import test_colrs_layout as C
import test_rowio_layout as R

# (L, rows per CTA, tile width, threads)
ROWS = [(128, 4, 2, 128), (256, 4, 2, 128), (512, 4, 2, 256), (1024, 2, 2, 256), (1024, 4, 2, 512),
        (2048, 2, 1, 512), (2048, 8, 1, 512), (4096, 4, 2, 512)]


# the same of FP64 tiling 0
ROWS64 = [(256, 2, 1, 128), (512, 1, 1, 128), (1024, 2, 1, 256), (2048, 1, 1, 256)]


@pytest.mark.parametrize("f64,L,RR,W,NT", [(False, *r) for r in ROWS] + [(True, *r) for r in ROWS64])
def test_row_tiles(f64, L, RR, W, NT, monkeypatch):
    monkeypatch.setattr(R, "cfg", lambda f, l, v: (l // 2, RR, W, NT, R.seq_stride(l // 2)))
    assert L % RR == 0 and (L <= NT or L % NT == 0)
    R.test_fixed_copy_offsets_equal_the_general_map(f64, L, 0)
    R.test_general_map_stays_in_the_tile_and_the_rows(f64, L, 0)


def test_two_column_ctas_at_2048(monkeypatch):
    monkeypatch.setattr(C, "cfg", lambda L, W: (2, 256, True))
    C.test_shared_memory_accesses_are_bank_conflict_free(2048, 2)
    C.test_global_accesses_of_a_warp_are_contiguous_runs(2048, 2)
    C.test_column_pass_addresses_stay_inside_their_buffers(2048, 2)

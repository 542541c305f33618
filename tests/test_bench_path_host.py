"""The bench's description of the TRMM path names what the library's automatic rule runs:
one launch by rows from order 256 on (six-term split), the thin product up to 32
right-hand sides, 64-row leaves below."""
import bench


def test_trmm_path():
    for k, n, what in ((16384, 16384, "TRMM in one launch by 128-row tiles"),
                       (256, 100, "TRMM in one launch by 128-row tiles"), (255, 100, "TRMM 64"),
                       (512, 32, "TRMM as one thin product")):
        assert what in bench.auto_path_desc(k, n), (k, n)
    bench.SPLIT_TERMS, kept = 3, bench.SPLIT_TERMS
    try:
        assert "1024-row diagonal blocks" in bench.auto_path_desc(16384, 16384)
    finally:
        bench.SPLIT_TERMS = kept

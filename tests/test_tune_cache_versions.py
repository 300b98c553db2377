"""Versions of the tuning cache's lines: FP64 shapes tuned for the kernels before block
fixed point are not used for the present ones."""
from paper_1901_02211_gb300 import smpq as S

DEV, DIMS = "NVIDIA GB300/152sm", (8, 8, 8, 16)


def test_old_fp64_lines_are_ignored(tmp_path):
    path = str(tmp_path / "tune.txt")
    line = "|%s|8 8 8 16|72|%d|24 8 4 1 0|1.0\n"
    with open(path, "w") as f:
        for prec in (S.SMPQ_FP64, S.SMPQ_FP32, S.SMPQ_MIXED):
            f.write("smpq-tune-2" + line % (DEV, prec))
    assert S.smpq_tune_cache_lookup(path, DEV, DIMS, 72, S.SMPQ_FP64) is None
    for prec in (S.SMPQ_FP32, S.SMPQ_MIXED):
        assert S.smpq_tune_cache_lookup(path, DEV, DIMS, 72, prec) == (24, 8, 4, 1, 0)
    S.smpq_tune_cache_store(path, DEV, DIMS, 72, S.SMPQ_FP64, (24, 2, 4, 1, 0), 2.0)
    assert S.smpq_tune_cache_lookup(path, DEV, DIMS, 72, S.SMPQ_FP64) == (24, 2, 4, 1, 0)

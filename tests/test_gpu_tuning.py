"""The autotuner's table: every bucket, caps up to the kernel's own, read back as written."""
import os

import pytest

from paper_2605_27515_gb300 import qlb as Q

CAPS = {1, 2, 4, 8, 16, 32, 64}


def _table(path):
    with open(path) as f:
        rows = [tuple(int(x) for x in line.split()) for line in f if not line.startswith("#")]
    return {(m, K): cap for m, K, cap in rows}


def _check(table):
    assert set(table) == {(m, K) for m in (32, 64, 128, 256) for K in (256, 1024, 4096)}
    assert set(table.values()) <= CAPS
    # 256 rows make more tiles of 16 than half the grid: no cap above 2 changes anything, so the
    # kernel's own is kept, and the short buckets split into fewer than 16 parts whatever the cap
    assert max(table.values()) == 64


def test_committed_table(repo_root):
    _check(_table(os.path.join(repo_root, "paper_2605_27515_gb300", "tuning", "gram_splitk_gb300.txt")))


@pytest.mark.gpu
def test_autotune(tmp_path):
    ctx = Q.Ctx(device=0)
    path = str(tmp_path / "table.txt")
    ctx.autotune(path)
    _check(_table(path))
    ctx.load_tuning(path)
    ctx.close()

"""The traffic records' guard follows the device code and nothing else: a change
of host code or of a comment leaves the hash, one of a kernel does not."""

import os
import shutil
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

DSLASH = "paper_1612_02750_gb300/csrc/dslash.cu"
KERNELS = "paper_1612_02750_gb300/csrc/qex_kernels.cuh"
PARAMS = "paper_1612_02750_gb300/csrc/qex_dslash_params.cuh"


@pytest.fixture
def edited(tmp_path, monkeypatch):
    """The Dslash hash of a copy of the sources with one edit."""
    import bench

    monkeypatch.setattr(bench, "ROOT", str(tmp_path))

    def hash_with(rel=None, old=None, new=None):
        for f in bench.DSLASH_FILES:
            os.makedirs(os.path.dirname(tmp_path / f), exist_ok=True)
            shutil.copy(os.path.join(ROOT, f), tmp_path / f)
        if rel:
            text = (tmp_path / rel).read_text()
            assert text.count(old) >= 1, old
            (tmp_path / rel).write_text(text.replace(old, new))
        return bench.kernel_source_hash()

    return hash_with


@pytest.mark.parametrize("rel,old,new", [
    (DSLASH, "if (persistent < full) *grid = persistent;", "if (persistent < full) *grid = persistent + 1;"),
    (DSLASH, 'set_error("the residual epilogue is FP64 only");', 'set_error("FP64 only");'),
    (DSLASH, "// Shape of a Dslash launch", "// The shape of a launch"),
    (PARAMS, "if (fp64) return naik ? 340000 : 107000;", "if (fp64) return 0;"),
    (KERNELS, "qex_status launch_dslash(", "qex_status  launch_dslash("),
])
def test_host_code_and_comments_leave_the_hash(edited, rel, old, new):
    assert edited(rel, old, new) == edited()


@pytest.mark.parametrize("rel,old,new", [
    (DSLASH, "pdl_wait();", "pdl_wait(); pdl_wait();"),
    (DSLASH, "part += d;", "part -= d;"),
    (PARAMS, "S->pAp = tot;", "S->pAp = 2 * tot;"),
    (KERNELS, "S->true_rr = tot;", "S->true_rr = -tot;"),
    (KERNELS, "#define QEX_GRAPH_UNROLL 8", "#define QEX_GRAPH_UNROLL 4"),
])
def test_device_code_changes_the_hash(edited, rel, old, new):
    assert edited(rel, old, new) != edited()

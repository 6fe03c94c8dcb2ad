"""The autotuner on both sides of the size below which the Dslash has one shape."""

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1612_02750_gb300 import build

    build.build()
    import paper_1612_02750_gb300 as mod

    mod.load()
    return mod


@pytest.mark.parametrize("prec,naik", [("f64", False), ("f64", True), ("f32", False), ("f32r12", True),
                                       ("f32r12h", False), ("f32s16", True)])
def test_one_shape_is_not_timed(q, monkeypatch, prec, naik):
    """The first call on a small lattice launches its own kernel and no other,
    and qex_tune keeps the compiled Dslash shape, timing the vector update alone
    (at most 2 + 3 + 3 x 50 launches each of 4 grids)."""
    monkeypatch.delenv("QEX_TUNE", raising=False)
    monkeypatch.delenv("QEX_TUNE_CACHE", raising=False)
    lat = q.Lattice((10, 6, 4, 8))  # a size no other test uses: not in the process's cache
    fat = q.empty_links(lat, prec).zero_()
    lng = q.empty_links(lat, q.qex_long_links_prec(prec)).zero_() if naik else None
    x = q.empty_field(lat, prec).zero_()
    default = {k: v for k, v in q.qex_tune_info(lat, prec, naik).items() if k != "source"}
    n = q.qex_launch_count()
    q.qex_dslash(lat, prec, fat, lng, -1.0 / 24.0, 1, x)
    assert q.qex_launch_count() - n == 1
    q.qex_tune(lat, prec, fat, lng)
    assert q.qex_launch_count() - n <= 1 + 4 * (2 + 3 + 3 * 50)
    info = q.qex_tune_info(lat, prec, naik)
    assert info["source"] == "measured"
    for k in ("dslash_block", "reduce_block", "reduce_blocks_per_sm", "dslash_waves"):
        assert info[k] == default[k], k

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


# the smallest lattices of each format whose Dslash follows the measured shape, and a larger one
SHAPED = [("f64", False, (22, 22, 22, 22)), ("f64", True, (24, 24, 26, 48)), ("f32", False, (18, 16, 20, 20)),
          ("f32", True, (26, 26, 26, 28)), ("f32r12", False, (16, 16, 16, 22)), ("f32r12", True, (32, 32, 32, 38)),
          ("f32r12h", False, (12, 14, 18, 20)), ("f32r12h", True, (16, 16, 16, 18)),
          ("f32s16", False, (12, 14, 18, 20)), ("f32s16", True, (16, 16, 16, 18)), ("f32r12h", False, (20, 22, 24, 26))]


@pytest.mark.parametrize("prec,naik,dims", SHAPED)
def test_every_shape_keeps_dslash_bits(q, prec, naik, dims):
    """Plain and normal-operator Dslash give the same fields with the compiled
    shape and with others of the tuner's candidates, set by name."""
    import torch

    lx, ly, lz, lt = dims
    g = torch.Generator(device="cuda")
    g.manual_seed(31)
    lat = q.Lattice(dims)
    u = torch.view_as_complex(torch.rand((lt, lz, ly, lx, 4, 3, 3, 2), generator=g, device="cuda", dtype=torch.float64)
                              - 0.5)
    fat = q.qex_pack_links(lat, prec, u)
    lng = q.qex_pack_links(lat, q.qex_long_links_prec(prec), u) if naik else None
    x = q.empty_field(lat, prec).normal_(generator=g)
    c3 = -1.0 / 24.0 if naik else 0.0
    ref = None
    for block, red, per_sm, waves in ((256, 256, 2, 0), (64, 64, 8, 0), (128, 256, 0, 2), (256, 128, 4, 2)):
        q.qex_tune_set(lat, prec, naik, dslash_block=block, reduce_block=red, reduce_blocks_per_sm=per_sm,
                       dslash_waves=waves)
        got = q.qex_dslash(lat, prec, fat, lng, c3, 1, x), q.qex_normal_op(lat, prec, fat, lng, c3, 0.1, x)
        ref = ref or got
        assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1]), (block, red, per_sm, waves)

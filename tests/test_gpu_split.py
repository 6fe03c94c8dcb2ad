"""The Dslash of small lattices, whose directions run on four threads a site:
both sides of the size where it ends, and ragged tails, against the multi-RHS
kernel with one right-hand side (one thread a site at every size)."""

import pytest

pytestmark = pytest.mark.gpu

C3 = -1.0 / 24.0
# the two kernels sum a site's 48 or 96 products in another order: a few ulp
TOL = {"f64": 1e-15, "f32": 1e-6, "f32r12": 1e-6, "f32r12h": 1e-6, "f32s16": 1e-6}


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


CASES = [("f64", False, (20, 22, 22, 22)), ("f64", False, (22, 22, 22, 22)),
         ("f64", True, (24, 24, 24, 48)), ("f64", True, (24, 24, 26, 48)),
         ("f32", False, (16, 16, 20, 20)), ("f32", False, (18, 16, 20, 20)),
         ("f32", True, (26, 26, 26, 26)), ("f32", True, (26, 26, 26, 28)),
         ("f32r12", False, (16, 16, 16, 20)), ("f32r12", False, (16, 16, 16, 22)),
         ("f32r12", True, (32, 32, 32, 36)), ("f32r12", True, (32, 32, 32, 38)),
         ("f32r12h", False, (10, 14, 18, 22)), ("f32r12h", False, (12, 14, 18, 20)),
         ("f32r12h", True, (16, 16, 16, 16)), ("f32r12h", True, (16, 16, 16, 18)),
         ("f32s16", False, (10, 14, 18, 22)), ("f32s16", False, (12, 14, 18, 20)),
         ("f32s16", True, (16, 16, 16, 16)), ("f32s16", True, (16, 16, 16, 18))]


@pytest.mark.parametrize("prec,naik,dims", CASES + [(p, False, d) for p in TOL for d in ((2, 2, 2, 2), (6, 2, 10, 2))]
                         + [(p, True, (6, 4, 10, 4)) for p in TOL])
def test_split_matches_one_thread_a_site(q, prec, naik, dims):
    import torch

    lx, ly, lz, lt = dims
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    lat = q.Lattice(dims)
    shape = (lt, lz, ly, lx, 4, 3, 3, 2)
    u = torch.view_as_complex(torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) - 0.5)
    fat = q.qex_pack_links(lat, prec, u)
    lng = q.qex_pack_links(lat, q.qex_long_links_prec(prec), u.conj().resolve_conj().contiguous()) if naik else None
    for p in (0, 1):
        x = q.empty_field(lat, prec).normal_(generator=g)
        got = q.qex_dslash(lat, prec, fat, lng, C3, p, x)
        ref = q.qex_dslash_mrhs(lat, prec, fat, lng, C3, p, 1, x)
        assert torch.linalg.norm(got - ref).item() <= TOL[prec] * torch.linalg.norm(ref).item(), p
        if p == 0:
            y = q.empty_field(lat, prec).normal_(generator=g)
            tmp = q.empty_field(lat, prec)
            out = q.qex_normal_op(lat, prec, fat, lng, C3, 0.3, y, None, tmp)
            ref = 0.09 * y - q.qex_dslash_mrhs(lat, prec, fat, lng, C3, 0, 1, tmp)
            assert torch.linalg.norm(out - ref).item() <= TOL[prec] * torch.linalg.norm(ref).item()

"""The multi-RHS Dslash by its three paths (two fields a thread, four with the
hops staged in shared memory, four with direct loads): both sides of the sizes
where they meet, group tails and ragged lattices, each field against the same
field alone."""

import pytest

pytestmark = pytest.mark.gpu

C3 = -1.0 / 24.0


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


# 152 SMs: 12^4 is 41 blocks of sites, (10, 14, 18, 22) 109
CASES = [(p, n, d, r) for p in ("f32", "f32r12", "f32r12h", "f32s16") for n in (False, True)
         for d, r in (((12, 12, 12, 12), 6), ((12, 12, 12, 12), 7), ((12, 12, 12, 12), 13),
                      ((10, 14, 18, 22), 3), ((10, 14, 18, 22), 9), ((10, 14, 18, 22), 11))]
CASES += [("f32", False, (16, 16, 18, 18), 7), ("f32", False, (16, 18, 18, 18), 7),
          ("f32r12", False, (18, 18, 20, 20), 8), ("f32r12h", False, (20, 22, 24, 24), 5),
          ("f32r12h", False, (20, 24, 24, 24), 7), ("f32s16", True, (18, 18, 18, 18), 10),
          ("f64", False, (12, 12, 12, 12), 5), ("f64", True, (4, 6, 4, 10), 64), ("f32r12", True, (4, 6, 4, 10), 63)]


@pytest.mark.parametrize("prec,naik,dims,nrhs", CASES)
def test_paths_match_one_field(q, prec, naik, dims, nrhs):
    import torch

    lx, ly, lz, lt = dims
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    lat = q.Lattice(dims)
    shape = (lt, lz, ly, lx, 4, 3, 3, 2)
    u = torch.view_as_complex(torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) - 0.5)
    fat = q.qex_pack_links(lat, prec, u)
    lng = q.qex_pack_links(lat, q.qex_long_links_prec(prec), u.conj().resolve_conj().contiguous()) if naik else None
    x = torch.cat([q.empty_field(lat, prec) for _ in range(nrhs)]).normal_(generator=g)
    # every path does a field's arithmetic in the same order; a few ulp, should a
    # product be contracted differently
    tol = 1e-15 if prec == "f64" else 1e-6
    for p in (0, 1):
        got = q.qex_dslash_mrhs(lat, prec, fat, lng, C3, p, nrhs, x)
        for a, b in zip(got.chunk(nrhs), x.chunk(nrhs)):
            ref = q.qex_dslash_mrhs(lat, prec, fat, lng, C3, p, 1, b.clone())
            assert torch.linalg.norm(a - ref).item() <= tol * torch.linalg.norm(ref).item(), p

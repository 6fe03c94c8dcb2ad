"""The persistent CG kernel where a thread has more than one site, and its
lattices by the other route: solves of every inner precision, ragged last
rounds among them, against the graph solve asked for by name."""

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


# One block of 512 threads an SM takes 128 sites at once in FP32, two of 256 take 64 each in FP64, 19,456 on 152
# SMs: the larger lattices go round more than once, and their last round is not full.
CASES = [(p, n, d) for p in ("f64", "f32", "f32r12", "f32r12h", "f32s16") for n in (False, True)
         for d in ((8, 8, 8, 8), (6, 4, 10, 4), (14, 14, 14, 16))]
CASES += [("f64", False, (16, 16, 16, 16)), ("f64", True, (18, 14, 16, 10)), ("f32", True, (20, 20, 22, 22)),
          ("f32r12", False, (18, 20, 16, 22)), ("f32r12h", True, (16, 16, 16, 22)), ("f32s16", False, (16, 18, 14, 14))]


@pytest.mark.parametrize("inner,naik,dims", CASES)
def test_fused_matches_graph(q, monkeypatch, inner, naik, dims):
    """A few iterations and a whole solve by both routes.  They differ in the
    order of the sums alone: six iterations by a few hundred roundings of the
    inner precision.  Solutions of true residual 1e-10 (by the library's FP64
    operator) differ by at most 2e-10 (m^2 + |D|^2) / m^2 of their norm; Haar
    links at m = 0.5, long links of norm 3: |D| <= 8 (1 + 3 / 24), 6.5e-8."""
    import torch

    m = 0.5
    lx, ly, lz, lt = dims
    g = torch.Generator(device="cuda")
    g.manual_seed(17)
    shape = (lt, lz, ly, lx, 4, 3, 3, 2)

    def unitary():
        z = torch.view_as_complex(torch.randn(shape, generator=g, device="cuda", dtype=torch.float64))
        a = z[..., 0, :] / torch.linalg.norm(z[..., 0, :], dim=-1, keepdim=True)
        b = z[..., 1, :] - (a.conj() * z[..., 1, :]).sum(-1, keepdim=True) * a
        b = b / torch.linalg.norm(b, dim=-1, keepdim=True)
        return torch.stack([a, b, torch.linalg.cross(a, b, dim=-1).conj().resolve_conj()], dim=-2).contiguous()

    lat = q.Lattice(dims)
    fat64 = q.qex_pack_links(lat, "f64", unitary())
    lng64 = q.qex_pack_links(lat, "f64", 3.0 * unitary()) if naik else None
    fati, lngi = fat64, lng64
    if inner != "f64":
        fati = q.qex_convert_links(lat, "f64", fat64, inner)
        lngi = q.qex_convert_links(lat, "f64", lng64, q.qex_long_links_prec(inner)) if naik else None
    b = q.empty_field(lat, "f64").normal_(generator=g)
    c3 = C3 if naik else 0.0
    ulp = 1.1e-16 if inner == "f64" else 6e-8
    out = {}
    for mode in ("graph", "fused"):
        monkeypatch.setenv("QEX_CG_MODE", mode)
        few, x = torch.zeros_like(b), torch.zeros_like(b)
        st, stats = q.qex_cg(lat, inner, fat64, lng64, fati, lngi, c3, m, b, few, tol=1e-14, maxiter=6, delta=1e-12,
                             check=False)
        assert st == 5 and stats["iters"] == 6, (mode, st, stats)
        st, stats = q.qex_cg(lat, inner, fat64, lng64, fati, lngi, c3, m, b, x, tol=1e-10, delta=0.1, check=False)
        assert st == 0 and stats["converged"], (mode, st, stats)
        assert q.qex_true_residual(lat, fat64, lng64, c3, m, b, x) <= 1.01e-10
        out[mode] = few, x, stats["iters"]

    def diff(k):
        return (torch.linalg.norm(out["fused"][k] - out["graph"][k]) / torch.linalg.norm(out["graph"][k])).item()

    assert diff(0) <= 300 * ulp
    assert diff(1) <= 6.5e-8
    assert abs(out["fused"][2] - out["graph"][2]) <= max(3, out["graph"][2] // 50)

"""The solver's parity and edge cases by each of its routes: small lattices run the
fused kernel unless QEX_CG_MODE names another."""

import pytest
import test_gpu_force as force_tests
import test_gpu_parity as parity_tests
from test_gpu_parity import q  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["graph", "host"])
@pytest.mark.parametrize("naik", [False, True])
@pytest.mark.parametrize("inner", parity_tests.PRECS)
def test_cg_parity(q, oracle_mod, monkeypatch, mode, naik, inner):  # noqa: F811
    monkeypatch.setenv("QEX_CG_MODE", mode)
    parity_tests.test_cg_parity(q, oracle_mod, naik, inner)


@pytest.mark.parametrize("mode", ["graph", "host"])
def test_cg_edge_cases(q, oracle_mod, monkeypatch, mode):  # noqa: F811
    monkeypatch.setenv("QEX_CG_MODE", mode)
    parity_tests.test_cg_edge_cases(q, oracle_mod)


@pytest.mark.parametrize("mode", ["graph", "host"])
@pytest.mark.parametrize("inner", ["f64", "f32r12h"])
def test_cg_initial_guess(q, oracle_mod, monkeypatch, mode, inner):  # noqa: F811
    monkeypatch.setenv("QEX_CG_MODE", mode)
    parity_tests.test_cg_initial_guess_zero_and_one_site(q, oracle_mod, inner)


@pytest.mark.parametrize("inner,bound", [("f64", 1e-9), ("f32r12", 1e-7)])
def test_force_chain(q, oracle_mod, monkeypatch, inner, bound):  # noqa: F811
    monkeypatch.setenv("QEX_CG_MODE", "graph")
    force_tests.test_force_chain_matches_oracle(q, oracle_mod, inner, bound)

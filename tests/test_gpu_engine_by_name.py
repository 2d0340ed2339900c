"""The FP64 engine a caller names is the one that runs and is counted, and AUTO chooses by size."""
import numpy as np
import pytest

import oracle
import synthetic as syn

pytestmark = pytest.mark.gpu

SIMT, OZAKI = 1, 5


def _solve(pkg, p, engine):
    with pkg.Handle(precision="fp64", engine=engine, profile=True) as h:
        h.set_H(p.H0, p.H1)
        r = h.solve(p.beta, p.nocc, p.n)
        return r["P1"].cpu().numpy(), h.stats()


@pytest.mark.parametrize("N", [33, 200])
def test_named_fp64_engine(cuda, cdmpt_lib, N):
    """Sizes where AUTO takes DFMA. Both engines round each product at about 2^-50, so the results
    agree to the FP64 bar 1e-10."""
    p = syn.chain_1d(N, seed=2, beta=10.0, n=12)
    P, st = {}, {}
    for engine in ("auto", "simt", OZAKI):
        P[engine], st[engine] = _solve(cdmpt_lib, p, engine)
    assert st[OZAKI]["engine_launches"][SIMT] == 0 and st[OZAKI]["engine_launches"][OZAKI] > 0
    for engine in ("auto", "simt"):
        assert st[engine]["engine_launches"][OZAKI] == 0 and st[engine]["engine_launches"][SIMT] > 0
        assert oracle.rel_frobenius(P[engine], P[OZAKI]) < 1e-10


@pytest.mark.parametrize("N,full", [(200, False), (1152, True)])
def test_dfma_flop_count(cuda, cdmpt_lib, N, full):
    """DFMA products of symmetric results count N (N + 1) N flops on the 8 x 8 tiles, which compute
    half of them, and 2 N^3 where the 64 x 64 tiles compute all (18 x 18 tiles and more)."""
    p = syn.banded_random(N, bandwidth=8, seed=3, beta=4.0, n=8)
    with cdmpt_lib.Handle(precision="fp64", engine="simt", profile=True) as h:
        h.set_H(p.H0)
        h.solve(p.beta, p.nocc, p.n, want_P0=False)
        st = h.stats()
    each = st["gemm_flops"] / st["gemm_launches"]
    assert each == pytest.approx(2.0 * N ** 3 if full else float(N) * (N + 1) * N)

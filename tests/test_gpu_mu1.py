"""The chemical-potential response mu1 by itself, against the oracle.

mu1 averages the perturbation's level elements over the few levels near mu, so a dipole that is
large against H0 (a long chain, a wide band) turns errors of 1e-7 in the levels' weights into
errors of 1e-5 in mu1. Bar: 1e-6 of |(mu, mu1)|, the bar of the mixed precision, for FP32 and mixed;
energies are counted from two hoppings above the band's centre. Rounding Q = dP0/dmu to FP32 leaves
2^-24 h_rms / sqrt(N) / |(mu, mu1)|, below 1e-7 for all of these.
"""
import math

import numpy as np
import pytest

import oracle
import synthetic as syn

pytestmark = pytest.mark.gpu

_REF = {}


def _system(kind, N, seed, beta):
    f = syn.chain_1d if kind == "chain" else syn.banded_random
    p = f(N, seed=seed, beta=beta, n=14)
    p.H0 = p.H0 - 2.0 * np.eye(N)
    return p


def _reference(kind, N, seed, beta):
    key = (kind, N, seed, beta)
    if key not in _REF:
        p = _system(*key)
        _REF[key] = oracle.solve(p.H0, p.H1, p.beta, p.nocc, n=p.n, kind="rec")
    return _REF[key]


def _error(r, ref):
    return np.abs(np.asarray(r["mu1"]) - ref["mu1"]).max() / math.hypot(ref["mu"], *ref["mu1"])


@pytest.mark.parametrize("precision", ["fp32", "mixed"])
@pytest.mark.parametrize("kind,N,seed,beta", [("chain", 175, 6, 33.0), ("chain", 240, 4, 26.0),
                                              ("chain", 530, 2, 30.0), ("chain", 700, 10, 40.0),
                                              ("chain", 130, 11, 52.1), ("chain", 201, 25, 71.7),
                                              ("chain", 273, 39, 27.6),
                                              ("banded", 600, 8, 15.0), ("banded", 1200, 4, 27.0)])
def test_mu1_of_wide_perturbations(cuda, cdmpt_lib, kind, N, seed, beta, precision):
    p, ref = _system(kind, N, seed, beta), _reference(kind, N, seed, beta)
    with cdmpt_lib.Handle(precision=precision) as h:
        h.set_H(p.H0, p.H1)
        r = h.solve(p.beta, p.nocc, p.n)
        first = h.response1(p.H1)
    assert _error(r, ref) < 1e-6
    assert _error(first, ref) < 1e-6
    assert oracle.rel_frobenius(r["P1"][0].cpu().numpy(), ref["P1"][0]) < 1e-6


@pytest.mark.parametrize("kw", [dict(engine="3xtf32"), dict(ckpt_stride=4), dict(screen_tau=1e-9)])
def test_wide_perturbation_with_other_options(cuda, cdmpt_lib, kw):
    """Where the trajectory is not refined (an engine by name, checkpoints) or the products are
    screened, a wide perturbation's outputs keep the FP32 bar."""
    p, ref = _system("chain", 240, 4, 26.0), _reference("chain", 240, 4, 26.0)
    with cdmpt_lib.Handle(precision="fp32", **kw) as h:
        h.set_H(p.H0, p.H1)
        r = h.solve(p.beta, p.nocc, p.n)
    assert _error(r, ref) < 1e-5
    assert oracle.rel_frobenius(r["P1"][0].cpu().numpy(), ref["P1"][0]) < 1e-5


def test_dipole_counted_from_a_corner(cuda, cdmpt_lib):
    """H1 + c I has the response of H1 and mu1 + c: a lattice dipole counted from far outside the
    cell (c = 100) gives P1 within the FP32 bar, and mu1 - c as exactly as FP64 adds c."""
    p = syn.cubic_lattice((6, 7, 8), seed=5, beta=20.0, n=14)
    p.H0 = p.H0 - 2.0 * np.eye(p.N)
    ref = oracle.solve(p.H0, p.H1, p.beta, p.nocc, n=p.n, kind="rec")
    for precision in ("fp32", "mixed"):
        with cdmpt_lib.Handle(precision=precision) as h:
            h.set_H(p.H0, p.H1 + 100.0 * np.eye(p.N))
            r = h.solve(p.beta, p.nocc, p.n)
        assert oracle.rel_frobenius(r["P1"][0].cpu().numpy(), ref["P1"][0]) < 1e-5
        assert abs(r["mu1"][0] - 100.0 - ref["mu1"][0]) < 1e-6 * math.hypot(ref["mu"], ref["mu1"][0])

"""Batches at the edges of what the lockstep closed forms are fitted for."""
import math

import numpy as np
import pytest

import oracle
import synthetic as syn

pytestmark = pytest.mark.gpu


def _solve(pkg, probs, precision, n):
    b = pkg.Batch([p.N for p in probs], probs[0].H1.shape[0], precision=precision)
    try:
        b.set_H([p.H0 for p in probs], [p.H1 for p in probs], n)
        r = b.solve([p.beta for p in probs], [p.nocc for p in probs], n)
        return r, b.stats()
    finally:
        b.close()


@pytest.mark.parametrize("precision", ["fp32", "mixed"])
@pytest.mark.parametrize("width", [0.0, 1e-18, 1e-12, 1e-6])
def test_system_whose_levels_coincide(cuda, cdmpt_lib, width, precision):
    """Two levels `width` apart beside ordinary clusters: the shared polynomial shape is fitted to an
    interval of that width too. Bar: 1e-5, FP32's."""
    n = 10
    probs = syn.clusters(B=2, seed=77, sizes=[65, 200], beta=20.0, n=n)
    D = probs[0].H1.shape[0]
    H1 = np.zeros((D, 2, 2))
    H1[:, 0, 0], H1[:, 1, 1] = 0.5, -0.5
    probs.insert(1, syn.Problem("pair", np.array([[0.0, width], [width, 0.0]]), H1, nocc=1.0,
                                beta=20.0, n=n))
    r, st = _solve(cdmpt_lib, probs, precision, n)
    _, without = _solve(cdmpt_lib, [probs[0], probs[2]], precision, n)
    assert st["mu_iterations"] == without["mu_iterations"]
    assert st["kernel_launches"] < 1.2 * without["kernel_launches"]   # no fallback to CG
    for i, p in enumerate(probs):
        ref = oracle.solve(p.H0, p.H1, p.beta, p.nocc, n=n, kind="rec")
        assert oracle.rel_frobenius(r["P0"][i].cpu().numpy(), ref["P0"]) < 1e-5
        assert oracle.rel_frobenius(r["P1"][i].cpu().numpy(), ref["P1"]) < 1e-5


def test_mu1_of_wide_perturbations(cuda, cdmpt_lib):
    """Mixed batch of a wide band and long chains: mu1 to 1e-6 of |(mu, mu1)|, as single solves."""
    probs = [syn.banded_random(1200, seed=4, beta=27.0, n=14), syn.chain_1d(1477, 3, 13.0, 14),
             syn.chain_1d(240, 4, 26.0, 14)]
    for p in probs:
        p.H0 = p.H0 - 2.0 * np.eye(p.N)
    r, _ = _solve(cdmpt_lib, probs, "mixed", 14)
    for i, p in enumerate(probs):
        ref = oracle.solve(p.H0, p.H1, p.beta, p.nocc, n=14, kind="rec")
        err = np.abs(r["mu1"][i] - ref["mu1"]).max() / math.hypot(ref["mu"], *ref["mu1"])
        assert err < 1e-6, (i, err)


@pytest.mark.parametrize("precision", ["fp32", "mixed"])
@pytest.mark.parametrize("where", ["H0", "H1"])
def test_non_finite_system_is_refused(cuda, cdmpt_lib, where, precision):
    n = 10
    probs = syn.clusters(B=2, seed=78, sizes=[70, 150], beta=20.0, n=n)
    A = getattr(probs[1], where)
    A[..., 2, 5] = A[..., 5, 2] = np.nan
    with pytest.raises(cdmpt_lib.CdmptError) as e:
        _solve(cdmpt_lib, probs, precision, n)
    assert e.value.status == 4

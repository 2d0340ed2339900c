"""NaN and infinity in the inputs end with an error status, in every precision.

CG never meets its tolerance on a NaN, so such calls always ended with status 4; the closed forms
that stand in for it have no residual, and the digit products turn a NaN into some number. Sizes on
both sides of the FP64 line between DFMA tiles and digit products; the value sits off the diagonal,
where traces do not see it.
"""
import numpy as np
import pytest

import synthetic as syn

pytestmark = pytest.mark.gpu

PRECISIONS = ["fp64", "fp32", "mixed"]


def _problem(N):
    return syn.chain_1d(N, seed=3, beta=8.0, n=11)


def _spoiled(A, value):
    B = A.copy()
    B[..., 2, 5] = B[..., 5, 2] = value
    return B


def _refused(pkg, call):
    with pytest.raises(pkg.CdmptError) as e:
        call()
    assert e.value.status == 4


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("N", [40, 420])
@pytest.mark.parametrize("precision", PRECISIONS)
def test_solve_refuses(cuda, cdmpt_lib, precision, N, value):
    p = _problem(N)
    with cdmpt_lib.Handle(precision=precision) as h:
        h.set_H(p.H0, _spoiled(p.H1, value))
        _refused(cdmpt_lib, lambda: h.solve(p.beta, p.nocc, p.n))
        h.set_H(p.H0, p.H1)                       # the handle stays usable
        r = h.solve(p.beta, p.nocc, p.n)
        assert np.isfinite(r["mu1"]).all()


@pytest.mark.parametrize("N", [40, 420])
@pytest.mark.parametrize("precision", PRECISIONS)
def test_grand_canonical_solve_refuses(cuda, cdmpt_lib, precision, N):
    """A fixed mu: no occupation loop that a NaN could keep from converging."""
    p = _problem(N)
    with cdmpt_lib.Handle(precision=precision, grand_canonical=True, mu_guess=0.1) as h:
        h.set_H(_spoiled(p.H0, np.nan))
        _refused(cdmpt_lib, lambda: h.solve(p.beta, p.nocc, p.n))


@pytest.mark.parametrize("N", [40, 420])
@pytest.mark.parametrize("precision", PRECISIONS)
def test_derivatives_refuse(cuda, cdmpt_lib, precision, N):
    import torch
    p = _problem(N)
    with cdmpt_lib.Handle(precision=precision) as h:
        h.set_H(p.H0, p.H1)
        h.solve(p.beta, p.nocc, p.n)
        G0 = torch.from_numpy(_spoiled(np.eye(N), np.nan)).cuda()
        _refused(cdmpt_lib, lambda: h.vjp_P0(G0))
        _refused(cdmpt_lib, lambda: h.response1(_spoiled(p.H1, np.nan)))
        h.set_H_orders(_spoiled(p.H1, np.nan), None)
        _refused(cdmpt_lib, lambda: h.response2(want_grad=False))

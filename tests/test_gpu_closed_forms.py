"""The closed forms of the steps against conjugate gradients.

With an iteration cap below the polynomial's degree (18 at the FP64 tolerance) the solver takes
its CG path: the sweeps' saturated steps, the response, the adjoint, the second order and the
log-determinants. Both paths solve the same systems to a relative tolerance of 1e-13 per solve;
with at most 16 steps and a condition of 2 per step the results agree to 1e-11 in relative
Frobenius norm. Sizes: one tile, a remainder of one, the DFMA and the tensor-core products
(N = 450 is above their line), three directions.
"""
import numpy as np
import pytest

import oracle
import synthetic as syn

pytestmark = pytest.mark.gpu


def _run(pkg, p, cap, ckpt):
    import torch
    g = np.random.default_rng(5)
    G = g.standard_normal((p.N, p.N))
    with pkg.Handle(precision="fp64", cg_maxit=cap, ckpt_stride=ckpt) as h:
        h.set_H(p.H0, p.H1)
        r = h.solve(p.beta, p.nocc, p.n)
        out = {"P0": r["P0"], "P1": r["P1"], "vjp": h.vjp_P0(torch.from_numpy(0.5 * (G + G.T)).cuda()),
               "r1": h.response1(p.H1[:1])["P1"], "grad": h.response2()["grad"]}
        fe = h.free_energy()
        out["fe_grad"] = fe["grad"]
        it = h.stats()["cg_iterations_response"]
    return {k: v.cpu().numpy() for k, v in out.items()}, fe["omega"], it


@pytest.mark.parametrize("dims,ckpt", [((3, 4, 5), 0), ((5, 5, 5), 4), ((8, 8, 4), 0), ((5, 9, 10), 0)])
def test_closed_forms_match_cg(cuda, cdmpt_lib, dims, ckpt):
    p = syn.cubic_lattice(dims, seed=91, beta=12.0, n=13, directions="xyz")
    a, oa, ia = _run(cdmpt_lib, p, 200, ckpt)
    try:
        b, ob, ib = _run(cdmpt_lib, p, 17, ckpt)
    except cdmpt_lib.CdmptError as e:
        assert e.status == 4       # CG itself needs more than the cap: refused, as it should be
        pytest.skip("no CG result within 17 iterations")
    assert ia == 0 and ib > 0      # the second solve did take the CG path
    for k in a:
        assert oracle.rel_frobenius(a[k], b[k]) < 1e-11, k
    assert abs(oa - ob) < 1e-11 * abs(ob)


def test_batch_cap_takes_cg_and_agrees(cuda, cdmpt_lib):
    """FP32 batch, three uneven systems: a cap of 9 iterations (degree 10 at the FP32 tolerance)
    against the default, both within the FP32 bar 1e-5 of each other's P0 and P1."""
    probs = syn.clusters(B=3, seed=77, sizes=[65, 128, 200], n=12)
    out = []
    for cap in (200, 9):
        b = cdmpt_lib.Batch([q.N for q in probs], 3, precision="fp32", cg_maxit=cap)
        b.set_H([q.H0 for q in probs], [q.H1 for q in probs], 12)
        r = b.solve([q.beta for q in probs], [q.nocc for q in probs], 12)
        out.append(([x.cpu().numpy() for x in r["P0"]], [x.cpu().numpy() for x in r["P1"]],
                    b.stats()["cg_iterations_response"]))
        b.close()
    assert out[0][2] == 0 and out[1][2] > 0
    for i in range(3):
        assert oracle.rel_frobenius(out[0][0][i], out[1][0][i]) < 1e-5
        assert oracle.rel_frobenius(out[0][1][i], out[1][1][i]) < 1e-5

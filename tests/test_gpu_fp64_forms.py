"""FP64 solves at the edges of the product tiles, and the closed forms against CG above the DFMA line.

The symmetric products of both FP64 engines (8 x 8 DFMA tiles, 256 x 64 digit tiles) enumerate the
upper triangle and mirror it; a wrong tile, remainder or mirror shows in P0 and P1. Bar against the
oracle: 1e-10, the FP64 bar.

Closed forms against CG: a cap of 17 iterations lies below the bound of 18 that the closed forms
ask for at 1e-13, and CG itself needs at most 15, since at these temperatures |Z_k| stays below
0.9 (the bound (sqrt(1 + z^2) - 1) / (sqrt(1 + z^2) + 1) per iteration); so no case is left out.
Both solve to 1e-13 per step: 1e-11 after at most 13 steps of condition below 2.
"""
import numpy as np
import pytest

import oracle
import synthetic as syn

pytestmark = pytest.mark.gpu

OZAKI = 5


@pytest.mark.parametrize("engine", ["auto", "simt", OZAKI])
@pytest.mark.parametrize("N", [1, 2, 7, 8, 9, 63, 64, 65, 127, 129, 255, 257, 321, 324, 409, 449,
                               513])
def test_tile_edges(cuda, cdmpt_lib, N, engine):
    p = syn.chain_1d(N, seed=N, beta=6.0, n=10)
    p.nocc = max(0.5, N // 2)
    ref = oracle.solve(p.H0, p.H1, p.beta, p.nocc, n=p.n, kind="rec")
    with cdmpt_lib.Handle(precision="fp64", engine=engine) as h:
        h.set_H(p.H0, p.H1)
        r = h.solve(p.beta, p.nocc, p.n)
    P0 = r["P0"].cpu().numpy()
    assert np.array_equal(P0, P0.T)
    assert oracle.rel_frobenius(P0, ref["P0"]) < 1e-10
    if N > 1:   # the canonical response of one level is zero
        assert oracle.rel_frobenius(r["P1"][0].cpu().numpy(), ref["P1"][0]) < 1e-10


def _run(pkg, p, cap):
    import torch
    G = np.random.default_rng(5).standard_normal((p.N, p.N))
    with pkg.Handle(precision="fp64", cg_maxit=cap) as h:
        h.set_H(p.H0, p.H1)
        r = h.solve(p.beta, p.nocc, p.n)
        it = h.stats()["cg_iterations_response"]
        out = {"P0": r["P0"], "P1": r["P1"], "grad": h.response2()["grad"],
               "vjp": h.vjp_P0(torch.from_numpy(0.5 * (G + G.T)).cuda()),
               "r1": h.response1(p.H1[:1])["P1"]}
        fe = h.free_energy()
        out["fe_grad"] = fe["grad"]
    return {k: v.cpu().numpy() for k, v in out.items()}, fe["omega"], it


@pytest.mark.parametrize("dims,beta", [((3, 4, 5), 0.35), ((7, 7, 7), 0.2), ((5, 9, 10), 0.35),
                                       ((3, 9, 19), 0.25)])
def test_closed_forms_match_cg_above_the_dfma_line(cuda, cdmpt_lib, dims, beta):
    p = syn.cubic_lattice(dims, seed=91, beta=beta, n=13, directions="xy")
    a, oa, ia = _run(cdmpt_lib, p, 200)
    b, ob, ib = _run(cdmpt_lib, p, 17)
    assert ia == 0 and ib > 0      # the second solve did take the CG path
    for k in a:
        assert oracle.rel_frobenius(a[k], b[k]) < 1e-11, k
    assert abs(oa - ob) < 1e-11 * abs(ob)

"""Device memory that does not suffice ends with a status, and the handle stays usable.

The memory is taken by an allocation of the test's own; N = 1024, n = 14, FP32: 0.46 GB without the
low parts and digits of a refined trajectory (0.1 GB more), 60 MB for H0 and H1 and their copies.
"""
import contextlib
import math

import numpy as np
import pytest

import oracle
import synthetic as syn

pytestmark = pytest.mark.gpu

ERR_OOM = 7
MB = 1 << 20


@contextlib.contextmanager
def _leave(free_bytes):
    """Allocations that leave about free_bytes of the device, given back at the end."""
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held = []
    try:
        while torch.cuda.mem_get_info()[0] - free_bytes >= 4 * MB:
            rest = torch.cuda.mem_get_info()[0] - free_bytes
            held.append(torch.empty(min(rest, 64 << 30), dtype=torch.uint8, device="cuda"))
        yield
    finally:
        held.clear()
        torch.cuda.empty_cache()


@pytest.fixture
def chain():
    p = syn.chain_1d(1024, seed=8, beta=20.0, n=14)
    p.H0 = p.H0 - 2.0 * np.eye(p.N)
    return p, oracle.solve(p.H0, p.H1, p.beta, p.nocc, n=p.n, kind="rec")


def _check(r, p, ref, bar):
    assert oracle.rel_frobenius(r["P0"].cpu().numpy(), ref["P0"]) < bar
    assert oracle.rel_frobenius(r["P1"][0].cpu().numpy(), ref["P1"][0]) < bar
    assert abs(r["mu1"][0] - ref["mu1"][0]) < bar * math.hypot(ref["mu"], ref["mu1"][0])


@pytest.mark.parametrize("precision", ["fp64", "fp32", "mixed"])
def test_solve_after_out_of_memory(cuda, cdmpt_lib, chain, precision):
    p, ref = chain
    with cdmpt_lib.Handle(precision=precision) as h:
        h.set_H(p.H0, p.H1)
        with _leave(150 * MB):
            for _ in range(3):      # a second call must not take the first one's buffers as there
                with pytest.raises(cdmpt_lib.CdmptError) as e:
                    h.solve(p.beta, p.nocc, p.n, want_P0=False, want_P1=False)
                assert e.value.status == ERR_OOM
        _check(h.solve(p.beta, p.nocc, p.n), p, ref, 1e-5)


def test_fp32_without_room_for_the_refinement(cuda, cdmpt_lib, chain):
    """A wide perturbation where the plain solve fits and the refined one does not: the FP32 bar."""
    p, ref = chain
    import torch
    with cdmpt_lib.Handle(precision="fp32") as h:
        h.set_H(p.H0, p.H1)
        torch.cuda.synchronize()
        free0 = torch.cuda.mem_get_info()[0]
        with cdmpt_lib.Handle(precision="fp32", engine="3xtf32") as plain:
            plain.set_H(p.H0, p.H1)
            plain.solve(p.beta, p.nocc, p.n)
            need = free0 - torch.cuda.mem_get_info()[0]
        with cdmpt_lib.Handle(precision="mixed") as mixed:
            mixed.set_H(p.H0, p.H1)
            mixed.solve(p.beta, p.nocc, p.n)
            refined = free0 - torch.cuda.mem_get_info()[0]
        assert refined > need
        with _leave((need + refined) // 2):
            for _ in range(2):
                r = h.solve(p.beta, p.nocc, p.n)
                assert h.stats()["refine_passes"] == 0
                _check(r, p, ref, 1e-5)


def test_alternating_perturbations_keep_the_buffers(cuda, cdmpt_lib):
    """Solves with and without a wide perturbation on one handle: no reallocation in between."""
    import torch
    p = syn.chain_1d(512, seed=8, beta=20.0, n=14)
    p.H0 = p.H0 - 2.0 * np.eye(p.N)
    ref = oracle.solve(p.H0, p.H1, p.beta, p.nocc, n=p.n, kind="rec")
    narrow = 1e-3 * p.H1
    with cdmpt_lib.Handle(precision="fp32") as h:
        h.set_H(p.H0, p.H1)
        h.solve(p.beta, p.nocc, p.n)
        torch.cuda.synchronize()
        free0 = torch.cuda.mem_get_info()[0]
        for _ in range(2):
            h.set_H(p.H0, narrow)
            r = h.solve(p.beta, p.nocc, p.n)
            assert h.stats()["refine_passes"] == 0
            assert oracle.rel_frobenius(1e3 * r["P1"][0].cpu().numpy(), ref["P1"][0]) < 1e-5
            h.set_H(p.H0, p.H1)
            _check(h.solve(p.beta, p.nocc, p.n), p, ref, 1e-6)
            assert h.stats()["refine_passes"] > 0
        del r
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        assert torch.cuda.mem_get_info()[0] >= free0 - 16 * MB

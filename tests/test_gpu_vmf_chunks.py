"""The adjoint's pixel pass with its seeds in chunks, at the sizes where the
split ends (below 256 seeds one chunk, chunks of a multiple of 64, a shorter
last one), against the FP64 reference.
Tolerance: the adjoint's 1e-4 relative L2 of its other tests.
"""
import pytest
import torch

import synth
from oracle import vmf_ref

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return ((a.double().cpu() - b).norm() / b.norm()).item()


@pytest.mark.parametrize("N,M", [(1, 600), (255, 255), (257, 256), (700, 385), (1500, 513), (300, 1000)])
def test_seed_chunks(ms_lib, N, M):
    prob = synth.vmf_problem_c5(seed=N, N=max(N, M), M=M, K=8)
    P, X0 = torch.from_numpy(prob["P"])[:N].contiguous(), torch.from_numpy(prob["X0"])
    G = torch.randn(M, 16, generator=torch.Generator().manual_seed(3))
    dP, dX0 = ms_lib.ms_vmf_backward(P.cuda(), X0.cuda(), 20.0, 2, G.cuda())
    _, rP, rX = vmf_ref.vmf_vjp(P.double(), X0.double(), 20.0, 2, G.double())
    assert _rel(dP, rP) <= 1e-4
    # one pixel: every x' is that pixel and dX0 is rounding of zero
    assert N == 1 or _rel(dX0, rX) <= 1e-4

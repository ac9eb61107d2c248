"""Device memory that holds the matrices of a binary64 solve but not the digit planes of its products:
the solve runs without them. And a solve that is refused for lack of memory leaves nothing behind
for the next one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import ksinputs  # noqa: E402
import paper_1705_11191_gb300 as egb  # noqa: E402

MB = 1 << 20


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


class Filled:
    """All free device memory but `leave` bytes taken, in pieces."""

    def __init__(self, leave):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.held = []
        for piece in (1 << 33, 1 << 30, 1 << 26, 1 << 22):
            while torch.cuda.mem_get_info()[0] - piece >= leave:
                self.held.append(torch.empty(piece, dtype=torch.uint8, device="cuda"))

    def release(self):
        self.held = []
        torch.cuda.empty_cache()


def test_binary64_solve_without_digit_planes():
    n = 2000
    p = ksinputs.cluster_problem(n, seed=11)
    H, S, P = dev(p.h), dev(p.s), torch.empty((n, n), dtype=torch.float64, device="cuda")
    C, g = torch.randn(n, n, dtype=torch.float64, device="cuda"), torch.randn(n, 300, dtype=torch.float64, device="cuda")
    ev = torch.linspace(-1, 1, n, dtype=torch.float64, device="cuda")
    torch.cuda.empty_cache()
    with egb.Handle(n, p.n_state, p.n_electron) as hd:
        hd.use_current_stream()
        free = torch.cuda.mem_get_info()[0]
        hd.dm_real(H, S, out=P)
        used = free - torch.cuda.mem_get_info()[0]
        ref, energy = P.clone(), hd.dm_real(H, S, out=P)[1]
        adj = hd.ev_adjoint(ev, C, None, g)
    planes = 16 * n * n  # at least
    mem = Filled(used - planes // 2)
    try:
        with egb.Handle(n, p.n_state, p.n_electron) as hd:
            hd.use_current_stream()
            _, e = hd.dm_real(H, S, out=P)
    finally:
        mem.release()
    assert torch.linalg.norm(P - ref) <= 1e-10 * torch.linalg.norm(ref)
    assert abs(e - energy) <= 1e-10 * abs(energy)
    # the adjoint: four n x 300 matrices, and what the call itself allocates (C^T, two n x n results)
    mem = Filled(3 * 8 * n * n + 5 * 8 * n * 300 + planes // 2)
    try:
        with egb.Handle(n, n, 0.0) as hd:
            hd.use_current_stream()
            got = hd.ev_adjoint(ev, C, None, g)
    finally:
        mem.release()
    for a, b in zip(got, adj):
        assert torch.linalg.norm(a - b) <= 1e-10 * torch.linalg.norm(b)


def test_a_refused_solve_leaves_no_error_behind():
    n = 1500
    p = ksinputs.cluster_problem(n, seed=12)
    H, S, P = dev(p.h), dev(p.s), torch.empty((n, n), dtype=torch.float64, device="cuda")
    with egb.Handle(n, p.n_state, p.n_electron) as hd:
        hd.use_current_stream()
        mem = Filled(30 * MB)
        try:
            with pytest.raises(egb.ElsiError):
                hd.dm_real(H, S, out=P)
        finally:
            mem.release()
        hd.dm_real(H, S, out=P)
    # Tr(P S) = the number of electrons
    assert abs(float((P * S).sum()) - p.n_electron) < 1e-8 * p.n_electron

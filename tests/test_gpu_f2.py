"""FP32 passes on pairs of lanes: every transform length on some axis and direction type against the oracle, with
pencil counts that are not multiples of four, and unaligned caller's arrays."""
import numpy as np
import pytest

import oracle
from oracle import CELL, NODE, EVEN as E, ODD as O, PER, UNB as U
from paper_2211_07777_gb300 import flups as F
from tests.gpu_util import cuda_solve, rel_linf

pytestmark = pytest.mark.gpu

LENGTHS = sorted({2 ** a * 3 ** b for a in range(13) for b in range(8) if 4 <= 2 ** a * 3 ** b <= 4096})
TYPES = {1: [(PER, PER)], 2: [(U, U), (E, E), (O, O)], 4: [(E, O), (O, E), (E, U), (U, O)]}
# FP32 rounding of six transforms of up to 4096 points (relative L_inf; white-noise input)
TOL = 1e-5


def _cases():
    out = []
    for i, P in enumerate(LENGTHS):
        for m in (1, 2, 4):
            if P % m or P // m < 4:
                continue
            axis = (i + m + 1) % 3
            others = [6, 9] if i % 2 else [4, 27]
            bcs = [(PER, PER), (E, O) if i % 3 else (U, U)]
            bcs.insert(axis, TYPES[m][(i + 1) % len(TYPES[m])])
            others.insert(axis, P // m)
            out.append((tuple(others), tuple(bcs), NODE if i % 4 == 1 else CELL, P, axis))
    return out


@pytest.mark.parametrize("n,bcs,center,P,axis", _cases(), ids=[f"{c[3]}-{'xyz'[c[4]]}-{c[0][c[4]]}" for c in _cases()])
def test_every_length_matches_the_oracle(n, bcs, center, P, axis):
    data = [v + (1 if center == NODE else 0) for v in n]
    rng = np.random.default_rng(P + axis)
    f = rng.standard_normal((data[2], data[1], data[0]))
    h = (1.0 / max(n),) * 3
    L = tuple(v * h[0] for v in n)
    kernel = "hej2" if any(U in b for b in bcs) else "spectral"
    ref = oracle.solve(f, oracle.Problem(bc=bcs, h=h, center=center, kernel=kernel))
    out, _ = cuda_solve(f, bcs, center, F.F32, kernel, L=L, h=h)
    assert rel_linf(out, ref) < TOL, rel_linf(out, ref)


@pytest.mark.parametrize("off", [0, 1, 2, 3])
@pytest.mark.parametrize("bcs", [((U, U), (E, O), (PER, PER)), ((PER, PER), (PER, PER), (E, E))], ids=["y-first", "z-first"])
def test_unaligned_arrays_give_the_same_bits(bcs, off):
    """The first direction runs along y or z, where groups of four x neighbours are one access if aligned."""
    import torch
    shape = (12, 16, 24)
    f = torch.from_numpy(np.random.default_rng(3).standard_normal(shape)).float().cuda()
    with F.Solver((24, 16, 12), bcs, prec=F.F32, green="hej2" if (U, U) in bcs else "spectral", h=(1 / 24,) * 3,
                  L=(1.0, 16 / 24, 0.5)) as s:
        want = torch.empty_like(f)
        s.solve(want, f)
        a = torch.empty(f.numel() + 8, device="cuda")[off:off + f.numel()].view(shape)
        b = torch.empty(f.numel() + 8, device="cuda")[off:off + f.numel()].view(shape)
        a.copy_(f)
        s.solve(b, a)
        torch.cuda.synchronize()
        assert torch.equal(b, want)


@pytest.mark.parametrize("bcs", [((E, E), (PER, PER), (PER, PER)), ((U, U), (O, O), (E, E)), ((PER, PER), (E, O), (U, U))],
                         ids=["x-first", "open-x", "y-first"])
@pytest.mark.parametrize("nx", [9, 18, 27])
def test_the_last_group_takes_nothing_from_the_padding(nx, bcs):
    """Odd row lengths in the workspace: their padding, NaN before the solve, lies beside the last packed pencils."""
    import torch
    n = (nx, 16, 12)
    f = np.random.default_rng(4).standard_normal(n[::-1])
    h = (1 / 27,) * 3
    L = tuple(v / 27 for v in n)
    kernel = "hej2" if any(U in b for b in bcs) else "spectral"
    ref = oracle.solve(f, oracle.Problem(bc=bcs, h=h, center=CELL, kernel=kernel))
    t = F.flups_init_topo(n, CELL, 1, F.F32)
    s = F.flups_init_solver(t, bcs, h, L, kernel)
    try:
        F.flups_setup_shared(s)
        ws = torch.full((F.flups_workspace_size(s) // 4,), float("nan"), device="cuda")
        rhs = torch.from_numpy(f).float().cuda()
        phi = torch.empty_like(rhs)
        F.flups_solve_ws(s, phi, rhs, ws)
        torch.cuda.synchronize()
        got = phi.double().cpu().numpy()
    finally:
        torch.cuda.synchronize()
        F.flups_cleanup(s)
        F.flups_topo_free(t)
    assert np.isfinite(got).all() and rel_linf(got, ref) < TOL, rel_linf(got, ref)

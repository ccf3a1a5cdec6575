"""FP64-class Poisson solves in 64-bit fixed point: every transform length on some axis and direction type
against the oracle, ragged tiles, and lanes of extreme, zero, infinite and NaN values."""
import numpy as np
import pytest

import oracle
from oracle import CELL, NODE, EVEN as E, ODD as O, PER, UNB as U
from paper_2211_07777_gb300 import flups as F
from paper_2211_07777_gb300 import serve
from tests.gpu_util import cuda_solve, rel_linf

pytestmark = pytest.mark.gpu

LENGTHS = sorted({2 ** a * 3 ** b for a in range(13) for b in range(8) if 4 <= 2 ** a * 3 ** b <= 4096})
# direction types by extension length over cells
TYPES = {1: [(PER, PER)], 2: [(U, U), (E, E), (O, O)], 4: [(E, O), (O, E), (E, U), (U, O)]}


def _cases():
    out = []
    for i, P in enumerate(LENGTHS):
        for m in (1, 2, 4):
            if P % m or P // m < 4:
                continue
            bc = TYPES[m][i % len(TYPES[m])]
            axis = (i + m) % 3
            # the other directions: enough points for the fixed-point passes, odd counts of pencils
            need = 70000 // P
            small = next(v for v in (8, 9, 12, 16, 18, 24, 27, 36, 54, 72, 96, 128, 162) if v * v >= need)
            bcs, n = [(PER, PER), (PER, PER)], [small, small]
            if i % 2:
                bcs[i % 3 == 0] = (U, U)
            bcs.insert(axis, bc)
            n.insert(axis, P // m)
            out.append((tuple(n), tuple(bcs), NODE if i % 3 == 1 else CELL, P, axis))
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
    out, _ = cuda_solve(f, bcs, center, F.F64, kernel, L=L, h=h)
    assert rel_linf(out, ref) < 1e-13, rel_linf(out, ref)


def _solve(f, prec=F.F64):
    return cuda_solve(f, ((U, U), (E, O), (PER, PER)), CELL, prec, "hej2", h=(1 / 48,) * 3,
                      L=tuple(v / 48 for v in (48, 32, 36)))[0]


def _field(seed=0):
    return np.random.default_rng(seed).standard_normal((36, 32, 48))


@pytest.mark.parametrize("scale", [2.0 ** -800, 2.0 ** -400, 2.0 ** 400, 2.0 ** 900])
def test_power_of_two_scales_are_exact(scale):
    a, b = _solve(_field()), _solve(_field() * scale)
    assert np.array_equal(a * scale, b)


def test_rows_of_very_different_size_keep_their_accuracy():
    f = _field(1) * 10.0 ** np.random.default_rng(2).integers(-12, 1, size=(36, 32, 1))
    ref = oracle.solve(f, oracle.Problem(bc=((U, U), (E, O), (PER, PER)), h=(1 / 48,) * 3, center=CELL, kernel="hej2"))
    assert rel_linf(_solve(f), ref) < 1e-14


def test_zero_field_gives_zero():
    assert np.array_equal(_solve(np.zeros((36, 32, 48))), np.zeros((36, 32, 48)))


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_input_makes_the_solution_nan(bad):
    f = _field()
    f[3, 4, 5] = bad
    assert np.isnan(_solve(f)).all()


# One-sign lanes: decoding errors with a preferred direction would add up in one mode (a peak plane over a positive
# background) or at one point (the inverse of a plane source's one-sign spectrum): 2048 half units of 2^-57 are 7e-15.
# The FP64 passes, and NumPy's, have errors up to 1e-15 here.
@pytest.mark.parametrize("face", [U, E], ids=["peak", "plane"])
def test_one_sign_lanes_gain_no_coherent_error(face):
    n, bcs, h = (2048, 8, 8), ((face, face), (PER, PER), (PER, PER)), (1 / 2048,) * 3
    f = np.zeros(n[::-1])
    if face == U:
        f += np.random.default_rng(8).random(2048) / 1024
        f[:, :, 700] = 1.0
    else:
        f[:, :, 0] = 1.0
    kernel = "hej2" if face == U else "spectral"
    L = (1.0, 8 / 2048, 8 / 2048)
    got = cuda_solve(f, bcs, CELL, F.F64, kernel, h=h, L=L)[0]
    ref = oracle.solve(f, oracle.Problem(bc=bcs, h=h, center=CELL, kernel=kernel))
    assert rel_linf(got, ref) < 1.5e-15, rel_linf(got, ref)


# A mean that the zero mode drops: the largest modes meet a factor of zero, and the solution's modes keep the accuracy of
# their own products.  (The FP64 passes have an error of 1e-15; products rounded at the scale of the largest mode times
# the largest factor gave 1.3e-13 in the complex fused pass and 1.5e-12 in the real one.)
@pytest.mark.parametrize("n,bcs", [((16, 16, 1024), ((PER, PER),) * 3), ((16, 16, 512), ((E, E),) * 3),
                                   ((1024, 8, 16), ((E, E), (PER, PER), (PER, PER)))], ids=["complex", "real", "x"])
def test_fields_with_a_mean(n, bcs):
    f = np.random.default_rng(8).random(n[::-1])
    h = (1.0 / max(n),) * 3
    got = cuda_solve(f, bcs, CELL, F.F64, "spectral", h=h, L=tuple(v * h[0] for v in n))[0]
    ref = oracle.solve(f, oracle.Problem(bc=bcs, h=h, center=CELL, kernel="spectral"))
    err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
    assert err < 6e-15, err


# Node-centred odd faces: the extension holds zeros there, whatever the caller's array has
@pytest.mark.parametrize("host", [False, True], ids=["device", "pinned"])
@pytest.mark.parametrize("bad", [1e20, np.nan])
@pytest.mark.parametrize("prec", [F.F64, F.F64E], ids=["f64", "f64e"])
@pytest.mark.parametrize("faces", [(O, O), (O, E), (E, O), (U, O), (O, U)], ids=["oo", "oe", "eo", "uo", "ou"])
def test_values_on_odd_node_faces_take_no_part(faces, prec, bad, host):
    import torch
    bcs, n = (faces, (PER, PER), (PER, PER)), (36, 32, 32)  # x goes first
    f = np.random.default_rng(6).standard_normal((n[2] + 1, n[1] + 1, n[0] + 1))
    zero, dirty = f.copy(), f.copy()
    for side in (0, 1):
        if faces[side] == O:
            zero[:, :, -side], dirty[:, :, -side] = 0.0, bad
    out = []
    with F.Solver((37, 33, 33), bcs, center=NODE, prec=prec, green="hej2" if U in faces else "spectral", h=(1 / 36,) * 3,
                  L=tuple(v / 36 for v in n)) as s:
        for a in (zero, dirty):
            if host:
                rhs = torch.from_numpy(a).pin_memory()
                phi = torch.empty_like(rhs).pin_memory()
                s.solve_host(phi, rhs)
            else:
                rhs = torch.from_numpy(a).cuda()
                phi = torch.empty_like(rhs)
                s.solve(phi, rhs)
            torch.cuda.synchronize()
            out.append(phi.cpu().numpy())
    assert np.isfinite(out[0]).all()
    assert np.array_equal(out[0], out[1])


def test_both_fp64_precisions_run_the_same_passes():
    assert np.array_equal(_solve(_field(), F.F64), _solve(_field(), F.F64E))


# both sides of the line between the warp engine and fixed point: extensions of 32768, 36864 and 46656 points
@pytest.mark.parametrize("prec", [F.F64, F.F64E])
@pytest.mark.parametrize("n", [(32, 32, 32), (32, 32, 36), (36, 36, 36), (8, 16, 512)])
def test_sizes_around_the_line_match_the_oracle(n, prec):
    f = np.random.default_rng(sum(n)).standard_normal(n[::-1])
    h = (1.0 / max(n),) * 3
    bcs, L = ((PER, PER),) * 3, tuple(v * h[0] for v in n)
    got = cuda_solve(f, bcs, CELL, prec, "spectral", h=h, L=L)[0]
    ref = oracle.solve(f, oracle.Problem(bc=bcs, h=h, center=CELL, kernel="spectral"))
    with F.Solver(n, bcs, L=L, h=h, prec=prec) as s:
        fixed = [x["fixed_point"] for x in s.features()]
    assert all(fixed) or not any(fixed)
    # FP64 and fixed point: six transforms' rounding, 1e-14; double-float passes: at most 15 butterfly levels of 2u,
    # u = 2^-48, per direction and way
    bound = 1e-14 if prec == F.F64 or fixed[0] else 6 * 15 * 2.0 ** -47
    assert np.linalg.norm(got - ref) < bound * np.linalg.norm(ref)


# Below the line, three components fill the device in short FP64 tiles along y (64 points between walls: runtime tiles)
@pytest.mark.parametrize("bcs", [((PER, PER),) * 3, ((PER, PER), (U, U), (PER, PER)), ((E, E), (O, O), (PER, PER))],
                         ids=["periodic", "open", "walls"])
@pytest.mark.parametrize("P", [32, 64])
def test_thin_vector_boxes_in_fp64_tiles(bcs, P):
    m = 2 if bcs[1][0] in (U, O) else 1
    n = (4, P // m, (4096 if bcs[0] == (E, E) else 8192) // P)  # 32768 points of the extension
    f = np.random.default_rng(P).standard_normal((3, *n[::-1]))
    h = (1.0 / max(n),) * 3
    L = tuple(v * h[0] for v in n)
    kernel = "hej2" if (U, U) in bcs else "spectral"
    got = cuda_solve(f, (bcs,) * 3, CELL, F.F64, kernel, h=h, L=L)[0]
    for c in range(3):
        ref = oracle.solve(f[c], oracle.Problem(bc=bcs, h=h, center=CELL, kernel=kernel))
        assert rel_linf(got[c], ref) < 1e-13


# FP64E Biot-Savart: the passes beside the curl write and read its double-float array (second direction complex, real
# with complex modes, real with real modes; a quarter-wave and a semi-open one)
@pytest.mark.parametrize("center", [CELL, NODE], ids=["cell", "node"])
@pytest.mark.parametrize("bcs", [((U, U), (U, U), (U, U)), ((E, E), (PER, PER), (U, U)), ((O, O), (E, O), (U, U)),
                                 ((E, U), (U, O), (E, E)), ((PER, PER), (PER, PER), (PER, PER))],
                         ids=["open", "wall-periodic", "walls", "semi", "periodic"])
def test_double_float_curl_between_fixed_point_passes(bcs, center):
    n = (36, 32, 48)
    data = [v + (1 if center == NODE else 0) for v in n]
    f = np.random.default_rng(12).standard_normal((3, data[2], data[1], data[0]))
    bc, h = serve.vector_bc(bcs), (1 / 48,) * 3
    L = tuple(v / 48 for v in n)
    kernel = "hej2" if any(U in b for b in bcs) else "spectral"
    got = {p: cuda_solve(f, bc, center, p, kernel, h=h, L=L, op=F.BIOT_SAVART)[0] for p in (F.F64, F.F64E)}
    # 15 butterfly levels of 2u, u = 2^-48, in the curl's two transforms
    assert np.linalg.norm(got[F.F64E] - got[F.F64]) < 2 * 15 * 2.0 ** -47 * np.linalg.norm(got[F.F64])
    f[1, 3, 4, 5] = np.nan
    assert np.isnan(cuda_solve(f, bc, center, F.F64E, kernel, h=h, L=L, op=F.BIOT_SAVART)[0]).any()


FIRST_PLANS = """
import sys, time
sys.path.insert(0, sys.argv[1])
import torch
from paper_2211_07777_gb300 import flups as F
def plan(n):
    t = time.perf_counter()
    F.Solver((n,) * 3, ((F.UNB, F.UNB),) * 3, prec=F.F64, green="hej2").close()
    return time.perf_counter() - t
torch.ones(1, device="cuda")
plan(32)
print(min(plan(n) for n in (64, 36, 48)))
"""


def test_the_first_plan_of_a_length_loads_its_kernels_quickly():
    """In a new process, after its first plan: the lengths' kernels load in 1 to 3 ms (20 ms and more with their line
    tables)."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", FIRST_PLANS, root], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert float(r.stdout) < 0.010, r.stdout

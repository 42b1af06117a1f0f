"""The FP64 form's fixed-point contractions (csrc/fixed.cuh) where they can go
wrong: ragged tiles of every element kind, weights whose common denominator
leaves the product range, states whose differences are subnormal before they
are aligned, and non-finite states; against the oracle at its FP64 bar (1e-12
of the summed-term scale, tests/test_gpu_parity.py)."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle as O
from paper_2609_07387_gb300 import inputs as I
from paper_2609_07387_gb300 import ucns

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _mesh(kind, n):
    nodes, cells, box = I.hex_lattice(n, jitter=0.1, seed=5)
    if kind == "tets":
        cells = I.split_tets(cells)
    if kind == "prisms":
        cells = I.split_prisms(cells)
    if kind == "pyramids":
        nodes, cells = I.split_pyramids(nodes, cells)
    if kind == "walls":
        box = np.array([box[0], box[1], 0.0])
    return nodes, cells, box


def _both(kind, n, order, scheme, Re=0.0, eps=1e-6, mach=0.5):
    nodes, cells, box = _mesh(kind, n)
    m = ucns.Mesh(nodes, cells, box, ucns.Params(order=order, scheme=scheme, Re=Re, Mach=mach, eps=eps))
    oc = O.Case(nodes, cells, box, O.Params(order=order, scheme=scheme, Re=Re, Mach=mach, eps=eps))
    return m, oc, I.noisy_state(nodes, cells, mach, 0.05, seed=6)


# cells stretched 100:1 (10:1 at P4, where the oracle rejects the stencils beyond),
# whose coefficients are scaled per axis
@pytest.mark.parametrize("order,stretch", [(2, 100.0), (3, 100.0), (4, 10.0)])
def test_stretched_cells(order, stretch):
    nodes, cells, box = I.hex_lattice((10, 9, 9), length=(1.0, stretch, 3.0), jitter=0.1, seed=5)
    p = dict(order=order, scheme=1, Re=1600.0, Mach=0.5)
    m, oc = ucns.Mesh(nodes, cells, box, ucns.Params(**p)), O.Case(nodes, cells, box, O.Params(**p))
    U = I.noisy_state(nodes, cells, 0.5, 0.05, seed=6)
    R, (Rc, S) = _residual(m, U), oc.residual_terms(U)
    err = np.abs(R - Rc).max(axis=1) / S.max(axis=1)
    print(order, err)
    assert np.all(err <= 1e-12)


def _residual(m, U):
    R = m.residual(torch.from_numpy(np.ascontiguousarray(m.to_internal(U))).cuda())
    return m.to_user(R.cpu().numpy())


# 210, 1050, 420, 1260 and 210 cells: the last 32-cell tile holds 18, 26, 4, 12 and 18 (810 and
# 900 at P3 and P4: 10 and 4);
# eps 1e-60 with a uniform z momentum and states scaled by 2^200 leave the range in
# which the weights share one denominator
@pytest.mark.parametrize("kind,n,order,scheme", [
    ("hexes", (5, 6, 7), 2, 1), ("hexes", (5, 6, 7), 2, 0), ("tets", (5, 5, 7), 2, 1), ("prisms", (5, 6, 7), 2, 1),
    ("pyramids", (5, 6, 7), 2, 1), ("walls", (5, 6, 7), 2, 1), ("hexes", (9, 9, 10), 3, 1), ("hexes", (9, 10, 10), 4, 1)])
@pytest.mark.parametrize("eps,scale", [(1e-6, 0), (1e-60, 0), (1e-6, 200)])
def test_residual_on_ragged_tiles(kind, n, order, scheme, eps, scale):
    m, oc, U = _both(kind, n, order, scheme, eps=eps)
    if eps < 1e-50:
        U[3] = 0.0
    U = U * 2.0 ** scale
    R, (Rc, S) = _residual(m, U), oc.residual_terms(U)
    err = np.abs(R - Rc).max(axis=1) / np.maximum(S.max(axis=1), 1e-300)
    print(kind, eps, scale, err)
    assert np.all(err <= 1e-12)


# The Euler residual with linear weights scales with the state; powers of two scale
# exactly through every operation, also where the state lies below the range in
# which differences are aligned directly (2^-962)
@pytest.mark.parametrize("order", [2, 3, 4])
@pytest.mark.parametrize("k", [-962, 600])
def test_power_of_two_states_scale_exactly(order, k):
    m, _, U = _both("hexes", (9, 9, 10), order, 0, mach=1.0)
    assert np.array_equal(_residual(m, U * 2.0 ** k), _residual(m, U) * 2.0 ** k)


# Cells of 2^40 with states of 2^-860: at P4 the quartic coefficients are subnormal (47
# bits of FP64's 53 left) and the zero ones have large offsets; the residual is the
# unit mesh's scaled, to the rounding of sums 1e3 times as large
@pytest.mark.parametrize("order", [2, 3, 4])
def test_large_cells_with_small_states(order):
    nodes, cells, box = I.hex_lattice((9, 9, 10), jitter=0.1, seed=5)
    U = I.noisy_state(nodes, cells, 1.0, 0.05, seed=6)
    R = []
    for L, u in ((0, 0), (40, -860)):
        m = ucns.Mesh(nodes * 2.0 ** L, cells, np.array(box) * 2.0 ** L, ucns.Params(order=order, scheme=0, Re=0.0, Mach=1.0))
        R.append(_residual(m, U * 2.0 ** u) * 2.0 ** (L - u))
    err = np.abs(R[1] - R[0]).max(axis=1) / np.abs(R[0]).max(axis=1)
    print(order, err)
    assert np.all(err <= 1e-12)


# Exact units beside round-off: differences just below a power of two, which round up
# to it (both signs, central and directional stencils)
@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("order", [2, 3, 4])
def test_units_beside_round_off(order, scheme):
    m, oc, U = _both("hexes", (9, 9, 10), order, scheme, mach=1.0)
    rng = np.random.default_rng(8)
    unit, tiny = rng.random(U.shape[1]) < 0.5, rng.choice([1e-18, -1e-18, 3e-18, -2e-19], size=U.shape[1])
    U[0], U[4] = 1.0, 10.0
    U[1] = np.where(unit, 1.0, tiny)
    U[2] = np.where(unit, -1.0, tiny)
    U[3] = np.where(unit, tiny, 0.5)
    R, (Rc, S) = _residual(m, U), oc.residual_terms(U)
    err = np.abs(R - Rc).max(axis=1) / S.max(axis=1)
    print(order, scheme, err)
    assert np.all(err <= 1e-12)


@pytest.mark.parametrize("order", [2, 3, 4])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_states_stay_visible(order, bad):
    m, oc, U = _both("hexes", (11, 11, 12), order, 0)
    U[1, 700] = bad
    assert np.array_equal(np.isfinite(_residual(m, U)), np.isfinite(oc.residual(U)))


# The FP64 form's tiles (35 KB a cell at P4, like the rows they are converted from) are
# uploaded in pieces: building a mesh takes the rows and little more of host memory
def test_host_memory_while_a_mesh_is_built():
    code = """
import numpy as np
from paper_2609_07387_gb300 import inputs as I, ucns
def peak():
    return next(int(x.split()[1]) for x in open("/proc/self/status") if x.startswith("VmHWM")) * 1024
def build(n):
    nodes, cells, box = I.hex_lattice(n, jitter=0.1, seed=5)
    return ucns.Mesh(nodes, cells, box, ucns.Params(order=4, scheme=1))
small = build(9)  # the CUDA context and the modules
before = peak()
build(24)
print(peak() - before)
"""
    out = subprocess.run([sys.executable, "-c", code], check=True, capture_output=True, text=True, timeout=300,
                         cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__)))).stdout
    # rows, matrices, stencils and face points in FP64
    rows = 24 ** 3 * (8 * (34 * 68 + 6 * 9 * 18 + 595 + 31) + 4 * (68 + 108) + 3 * 8 * 160)
    print(int(out) / rows)
    assert int(out) < 1.5 * rows

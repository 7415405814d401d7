"""GPU parity of the FP32 stage's two tile shapes at the sizes where they can go
wrong: meshes smaller than a block's first tile, ragged last tiles, and element
counts on both sides of the rule that picks the shape (a full round of
two-element tiles is 21,888 / 16,416 / 7,296 / 5,472 / 3,648 elements at N = 4 /
5 / 7 / 8 / 9 on 152 SMs)."""
import numpy as np
import pytest

import oracle as O
import paper_1211_0582_gb300 as dg
import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-5  # the FP32 bar: relative l2 error against the FP64 oracle


def rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


@pytest.mark.parametrize("N,n", [(N, n) for N in range(1, 10) for n in (1, 2)] +
                         [(1, 7), (2, 5), (3, 5), (6, 5), (4, 15), (5, 13), (7, 10), (8, 9), (9, 8), (5, 9), (8, 5)])
def test_shapes_match_the_oracle(N, n):
    VX, VY, VZ, EToV = W.kuhn_cube(n, jitter=0.1, seed=1)
    eps = W.element_eps(EToV.shape[0], seed=2)
    s = dg.Solver(N).upload(VX, VY, VZ, EToV, eps=eps)
    m = O.Mesh(N, VX, VY, VZ, EToV, eps=eps.astype(np.float64))
    u = np.random.default_rng(3).standard_normal(m.shape) + 2.0  # a constant part that the derivatives annihilate
    ud, rd = s.to_device(u), s.zeros()
    ud[:, :, s.Np:] = float("nan")  # padding entries are ignored
    ref = m.rhs(u)
    out = s.rhs(ud)
    assert not out[:, :, s.Np:].any()
    assert rel(s.from_device(out), ref) < TOL
    dt = 0.2 / n / max(N * N, 2.5)
    s.step(ud, rd, dt, 1)
    assert rel(s.from_device(ud), m.lserk(u, dt, 1)[0]) < TOL
    assert not ud[:, :, s.Np:].any() and not rd[:, :, s.Np:].any()


def test_nonfinite_values_stay_visible():
    # an infinity or a NaN at one node reaches its own element's right-hand side
    VX, VY, VZ, EToV = W.kuhn_cube(2, jitter=0.1, seed=1)
    s = dg.Solver(4).upload(VX, VY, VZ, EToV)
    for bad in (float("inf"), float("nan")):
        for node in (0, s.Np - 1):
            u = s.zeros()
            u[1, 7, node] = bad
            assert not s.rhs(u)[:, 7, :s.Np].isfinite().all()

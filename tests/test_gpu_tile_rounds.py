"""GPU parity of the stages on meshes of one to three rounds of tiles: full tiles
followed by a spread remainder, a block's second tile, and both sides of every rule
that picks a shape, the blocks per SM or half of the grid (element counts for the
152 SMs of a GB300).

Right-hand sides are compared with the FP64 oracle on the first and the last
elements and on a sample; steps with the scheme written out around the library's
own right-hand side."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_1211_0582_gb300 as dg
import workloads as W

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-5, "fp16x3": 1e-5, "bf16x3": 2e-4}
# five stages, each with the rounding of the state (2^-24) and of a right-hand side
# whose argument differs by that much (1e-6; 4e-5 for BF16x3), dt |A| about 1
STEP_TOL = {"fp32": 6e-6, "fp16x3": 6e-6, "bf16x3": 2e-4}
LSERK_A = (0.0, -567301805773.0 / 1357537059087.0, -2404267990393.0 / 2016746695238.0,
           -3550918686646.0 / 2091501179385.0, -1275806237668.0 / 842570457699.0)
LSERK_B = (1432997174477.0 / 9575080441755.0, 5161836677717.0 / 13612068292357.0,
           1720146321549.0 / 2090206949498.0, 3134564353537.0 / 4481467310338.0,
           2277821191437.0 / 14882151754819.0)


def first_elements(K):
    """The first K tetrahedra of a jittered cube (the faces that lose their neighbour become walls)."""
    n = int(np.ceil((K / 6) ** (1 / 3)))
    VX, VY, VZ, EToV = W.kuhn_cube(n, jitter=0.1, seed=1)
    EToV = EToV[:K]
    used, tets = np.unique(EToV, return_inverse=True)
    return n, (VX[used], VY[used], VZ[used], tets.reshape(-1, 4).astype(np.int32))


def check(precision, N, K):
    n, mesh = first_elements(K)
    eps = W.element_eps(K, seed=2)
    s = dg.Solver(N, precision=precision).upload(*mesh, eps=eps)
    m = O.Mesh(N, *mesh, eps=eps.astype(np.float64))
    u = np.random.default_rng(3).standard_normal(m.shape) + 2.0
    ud, rd = s.to_device(u), s.zeros()
    elems = np.unique(np.concatenate([np.arange(min(K, 24)), np.arange(max(0, K - 24), K),
                                      (W.uniform(21, 48) * K).astype(np.int64)]))
    got = s.from_device(s.rhs(ud))
    ref = m.rhs_subset(u, elems)
    assert np.linalg.norm(got[:, elems] - ref) < TOL[precision] * np.linalg.norm(ref)
    # every element: no tile left out, none written twice with another's values
    per_element = np.linalg.norm(got[:, elems] - ref, axis=(0, 2)) / np.linalg.norm(ref, axis=(0, 2))
    assert per_element.max() < 10 * TOL[precision]
    dt = 0.2 / n / max(N * N, 2.5)
    v, r = ud.clone(), torch.zeros_like(ud)
    for a, b in zip(LSERK_A, LSERK_B):
        r = (a * r.double() + dt * s.rhs(v).double()).float()
        v = (v.double() + b * r.double()).float()
    s.step(ud, rd, dt, 1)
    s.sync()
    assert float((ud - v).double().norm() / v.double().norm()) < STEP_TOL[precision]
    worst = (ud - v).double().norm(dim=(0, 2)) / v.double().norm(dim=(0, 2))
    assert float(worst.max()) < 10 * STEP_TOL[precision]
    assert not ud[:, :, s.Np:].any() and not rd[:, :, s.Np:].any()


# one-element shape: half of the blocks and all of them, past one round of all blocks (N <= 3, 6; at N = 3 the wide
# shape takes a round less from 14,593 to 15,200)
FP32 = [(1, 6080), (1, 6200), (1, 41154), (2, 9728), (2, 9800), (2, 20250), (3, 1368), (3, 1400), (3, 14592),
        (3, 14700), (3, 15300),
        (6, 1824), (6, 1900), (6, 4374),
        # N = 4: half and all of the blocks by turns, the one-element shape past a round, two rounds of the two-element one
        (4, 450), (4, 900), (4, 1300), (4, 3648), (4, 7400), (4, 24576),
        # N = 5: narrow, wide on half of the blocks, wide, narrow, wide, wide past a round, two rounds of the two-element one
        (5, 2432), (5, 2700), (5, 2800), (5, 3400), (5, 3700), (5, 5600), (5, 16464)]
# N >= 7: narrow, wide, a few elements past a round (narrow), past a round, two rounds of the two-element shape
for _N, _one, _wide, _two in ((7, 8, 16, 48), (8, 6, 12, 36), (9, 4, 8, 24)):
    FP32 += [(_N, 152 * _one), (_N, 152 * _one + 10), (_N, 152 * _wide), (_N, 152 * _wide + 30),
             (_N, 152 * _wide + 90), (_N, 152 * _two + 200)]


@pytest.mark.parametrize("N,K", FP32)
def test_fp32_rounds_match_the_oracle(N, K):
    check("fp32", N, K)


# at most a tile per SM, then up to four (N = 1) or two blocks per SM, then a second tile per block; N = 4, 5: half
# of the SMs, all, past a round; N = 6, 7: half up to 12 elements per tile
TC = [(1, 3040), (1, 3100), (1, 6100), (1, 9200), (1, 12500), (2, 60), (2, 3040), (2, 3100), (2, 6500), (3, 60),
      (3, 3040), (3, 3100), (3, 6500), (4, 900), (4, 1520), (4, 1600), (4, 3100), (5, 900), (5, 1520), (5, 1600),
      (5, 3100), (6, 912), (6, 930), (6, 3041), (7, 912), (7, 930), (7, 3041)]


@pytest.mark.parametrize("precision", ["fp16x3", "bf16x3"])
@pytest.mark.parametrize("N,K", TC)
def test_tensor_core_rounds_match_the_oracle(precision, N, K):
    check(precision, N, K)


@pytest.mark.parametrize("N,K", [(1, 3300), (2, 6500), (3, 700), (3, 6500), (4, 1300), (4, 3200), (5, 700), (5, 1300),
                                 (5, 2700), (5, 3100)])
def test_gradients_of_the_two_contexts_and_forms_agree(N, K):
    # the forward sweeps of an FP32 and of an FP16x3 context run different kernels (store forms), the reverse
    # sweeps two forms: whole rounds, a spread remainder, half of the blocks. Each is within 3e-5 of the exact
    # gradient (FP32 rounding over 10 stages of forward and reverse sweep)
    n, mesh = first_elements(K)
    eps = W.element_eps(K, seed=2)
    steps, dt = 2, 0.2 / n / max(N * N, 2.5)
    grads = []
    for precision, form in (("fp32", "cuda"), ("fp32", "tensor"), ("fp16x3", "tensor")):
        s = dg.Solver(N, precision=precision).upload(*mesh, eps=eps)
        s.set_adjoint_form(form)
        x, y, z = s.node_coords()
        u0 = s.to_device(W.cavity_mode(x, y, z, 0.0) + W.gaussian_pulse(x, y, z, seed=7)).requires_grad_()
        e = torch.as_tensor(eps, dtype=torch.float32, device="cuda").requires_grad_()
        recv = torch.as_tensor(np.unique((W.uniform(4, 200) * K * s.Np).astype(np.int64)), device="cuda")
        J = dg.ReceiverMisfit.apply(u0, e, s, recv, torch.zeros(steps, 3, recv.numel(), device="cuda"), dt, steps, 0,
                                    1.0)
        J.backward()
        grads.append((u0.grad.double(), e.grad.double()))
    for other in grads[1:]:
        for g, ref in zip(other, grads[0]):
            assert float((g - ref).norm() / ref.norm()) < 6e-5

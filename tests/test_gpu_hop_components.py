"""GPU: the FP64 hop component by component, on fields whose spins, colours or sites differ by orders of magnitude.

Bound: u = 2^-53 times 24 times the sum, over directions and colours, of |U| |h|, h the projected
neighbour.  FP64 sums stay within 15 u of it for a real part (1 for the projection, 6 for a
product's terms, 8 for the directions), which is 22 u for a complex number.  The fixed-point sums are
used where their error, 2^-56.1 of the block as a standard deviation, is at most 2 u of the sum.
"""
import numpy as np
import pytest
import torch

from lqhelp import Handle, dev, host
from paper_2001_07557_gb300 import inputs, lqcd
from test_gpu_halo import Slabs

pytestmark = pytest.mark.gpu

DIMS, V = (4, 6, 2, 4), 192
QUAD = np.clongdouble


def hop(U, psi, dag):
    """-1/2 times the hopping term in extended precision, and 1/2 the sums of |U| |h|."""
    ids = np.arange(V).reshape(DIMS[::-1])
    xs = np.meshgrid(*[np.arange(n) for n in DIMS[::-1]], indexing="ij")
    sig = np.array([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]])
    z, e = np.zeros((2, 2)), np.eye(2)
    gamma = [np.block([[z, -1j * s], [1j * s, z]]) for s in sig] + [np.block([[z, e], [e, z]])]
    U, psi = U.astype(QUAD), psi.astype(QUAD)
    out, size = np.zeros((V, 4, 3), QUAD), np.zeros((V, 4, 3), np.longdouble)
    for mu in range(4):
        ax = 3 - mu
        for bwd in (False, True):
            n = np.roll(ids, 1 if bwd else -1, ax).reshape(-1)
            edge = (xs[ax] == (0 if bwd else DIMS[mu] - 1)).reshape(-1)
            ph = np.where(edge & (mu == 3), -1, 1).reshape(-1, 1, 1)
            u = U[n, mu].conj().transpose(0, 2, 1) if bwd else U[:, mu]
            proj = np.eye(4) + (1 if bwd != dag else -1) * gamma[mu]
            h = sum(QUAD(1) * proj[:, t][None, :, None] * psi[n][:, None, t] for t in range(4))
            out += ph * sum(u[:, None, :, c] * h[:, :, None, c] for c in range(3))
            size += sum(np.abs(u)[:, None, :, c] * np.abs(h)[:, :, None, c] for c in range(3))
    return -out / 2, size / 2


def check(U, psi, U_prec=lqcd.LQ_F64):
    with Handle(DIMS, U, mass=-4.0, U_prec=U_prec) as H:
        for dag in (False, True):
            x = dev(psi)
            y = torch.empty_like(x)
            (lqcd.dslash_dag_apply if dag else lqcd.dslash_apply)(H.h, y, x, lqcd.LQ_F64, lqcd.LQ_FULL)
            want, size = hop(U, psi, dag)
            assert (np.abs(host(y) - want) <= 24 * 2.0 ** -53 * size).all()


def links(kind, seed=3700):
    if kind == "near 1":  # exp(i 1e-7 H): off the diagonal 1e-7
        return inputs.gauge_field(DIMS, "smooth", seed=seed, eps=1e-7)
    return inputs.gauge_field(DIMS, kind, seed=seed)


@pytest.mark.parametrize("kind", ["random", "smooth", "unit", "near 1"])
def test_dense_fields(kind):
    check(links(kind), inputs.gaussian_spinor(V, seed=3701))


@pytest.mark.parametrize("kind", ["random", "unit"])
@pytest.mark.parametrize("small", [0.1, 1e-2, 1e-4, 1e-8, 1e-12, 1e-30, 0.0])
def test_spins_of_different_size(kind, small):
    U = links(kind)
    for spin in range(4):
        psi = small * inputs.gaussian_spinor(V, seed=3702)
        psi[:, spin] = inputs.gaussian_spinor(V, seed=3703)[:, spin]
        check(U, psi)


@pytest.mark.parametrize("kind", ["unit", "near 1"])
@pytest.mark.parametrize("small", [0.1, 1e-2, 1e-4, 1e-8, 1e-12, 0.0])
def test_colours_of_different_size(kind, small):
    psi = inputs.gaussian_spinor(V, seed=3704)
    psi[..., 1] *= small
    psi[..., 2] *= small * small
    check(links(kind), psi)


@pytest.mark.parametrize("step", [0.5, 2, 8, 40])
def test_fields_that_fall_off(step):
    """exp(-step r) from one site, as propagators of heavy quarks do."""
    r = sum(np.minimum(x, n - x) for x, n in zip(np.meshgrid(*[np.arange(n) for n in DIMS[::-1]], indexing="ij"), DIMS[::-1]))
    psi = inputs.gaussian_spinor(V, seed=3705) * np.exp(-step * r.reshape(-1, 1, 1))
    for kind in ("random", "unit"):
        check(links(kind), psi)


def test_sources():
    """One spin and colour on every site (a volume source), on a time slice, and on one site."""
    for kind in ("random", "unit", "near 1"):
        U = links(kind)
        psi = np.zeros((V, 4, 3), complex)
        psi[:, 1, 2] = inputs.gaussian_spinor(V, seed=3706)[:, 0, 0]
        check(U, psi)
        psi[48:] = 0
        check(U, psi)
        psi[1:] = 0
        check(U, psi)


def test_links_given_in_fp32():
    for kind in ("random", "near 1"):
        U = links(kind).astype(np.complex64)
        psi = 1e-9 * inputs.gaussian_spinor(V, seed=3707)
        psi[:, 1] *= 1e9
        check(U, psi, lqcd.LQ_F32)


@pytest.mark.parametrize("projected", [False, True])
def test_slabs_with_ghost_faces(projected):
    """Sites that take the FP64 sums, and neighbours whose projection is exactly zero, come out of two time
    slabs bit for bit as out of one lattice."""
    dims, n = (4, 4, 4, 8), 512
    U = inputs.gauge_field(dims, "random", seed=3708)
    g = inputs.gaussian_spinor(n, seed=3709)
    small, plus, minus, mixed = g.copy(), g.copy(), g.copy(), g * np.exp(-np.arange(n) % 13)[:, None, None]
    small[:, [0, 2, 3]] *= 1e-8
    plus[:, 2:] = plus[:, :2]
    minus[:, 2:] = -minus[:, :2]
    point, wall = np.zeros_like(g), np.zeros_like(g)
    point[64 * 4 + 5, 1, 2] = 1
    wall[256:320, 3, 0] = g[256:320, 3, 0]
    S = Slabs(dims, 2, U, -4.0, (1, 1, 1, -1), lqcd.LQ_F64)
    try:
        with Handle(dims, U, mass=-4.0) as G:
            for psi in (small, plus, minus, mixed, point, wall):
                ins = S.scatter(psi)
                outs = [torch.zeros_like(i) for i in ins]
                for dag in (False, True):
                    S.hop(ins, outs, dagger=dag, projected=projected)
                    x = dev(psi)
                    y = torch.empty_like(x)
                    (lqcd.dslash_dag_apply if dag else lqcd.dslash_apply)(G.h, y, x, lqcd.LQ_F64, lqcd.LQ_FULL)
                    assert np.array_equal(S.gather(outs), host(y))
    finally:
        S.close()

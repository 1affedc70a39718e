"""The FP64 hopping term's block-integer arithmetic where its exponents matter: neighbours of very
different magnitudes, magnitudes outside the integer range (IEEE path), zeros, infinities and NaN.

The reference is the FP64 oracle. The bound is per (site, slice): both sides add 8 hops of sums of
at most 12 products of |U| <= 1 with |psi +- psi'| <= 2 max|psi|, each rounded to at most 2^-53 of
a partial sum, so they differ by less than 8 x 12 x 2 x 2^-53 x max|psi| over the neighbours of a
site (2.2e-14; the stored result's own rounding is far below it).
"""
import numpy as np
import pytest
import torch

from paper_2203_06777_gb300 import synth

pytestmark = pytest.mark.gpu

BC = (1, 1, 1, -1)
M5, MASS = 1.8, 0.01
BOUND = 8 * 12 * 2 * 2.0 ** -53
DIMS = (4, 6, 2, 4)


@pytest.fixture(scope="module")
def dwf():
    from paper_2203_06777_gb300 import dwf as mod

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    mod.load()
    return mod


def apply(dwf, U, psi, Ls, dag, c12=False):
    op = dwf.GridDWF(DIMS, Ls, M5, MASS, bc=BC, compress12=c12)
    op.set_gauge(torch.from_numpy(U).cuda())
    f = op.pack(torch.from_numpy(psi).cuda(), 0, dwf.FULL)
    return op.unpack(op.dhop(f, dwf.FULL, dag=dag)).cpu().numpy()


def neighbour_max(psi):
    """Largest magnitude over the neighbours of every (site, slice)."""
    m = np.abs(psi).max(axis=(-2, -1))
    return np.max([np.roll(m, d, ax) for ax in range(4) for d in (1, -1)], axis=0)


@pytest.mark.parametrize("Ls", [1, 3, 8, 10, 12, 16])
@pytest.mark.parametrize("spread", [0, 3, 40, 100])
def test_neighbours_of_different_magnitude(dwf, oracle_lib, Ls, spread):
    """Every (site, slice) scaled by a power of two from 2^-spread to 2^spread: the accumulator's
    exponent is raised by later hops, and small neighbours are shifted far below it."""
    U = synth.random_gauge(DIMS, seed=41)
    psi = synth.random_spinor(DIMS, Ls, seed=42)
    rng = np.random.default_rng(43)
    psi *= np.exp2(rng.integers(-spread, spread + 1, psi.shape[:5]))[..., None, None]
    psi[rng.random(psi.shape[:5]) < 0.2] = 0  # empty neighbours, first hops among them
    for dag in (False, True):
        ref = oracle_lib.dhop(DIMS, Ls, BC, U, psi, dag=dag)
        err = np.abs(apply(dwf, U, psi, Ls, dag) - ref).max(axis=(-2, -1))
        assert np.all(err <= BOUND * neighbour_max(psi))


@pytest.mark.parametrize("log2_psi,log2_u", [(-500, 0), (500, 0), (-1040, 0), (0, -450), (0, 450), (395, 390)])
def test_magnitudes_outside_the_integer_range(dwf, oracle_lib, log2_psi, log2_u):
    Ls = 4
    U = synth.random_gauge(DIMS, seed=44) * 2.0 ** log2_u
    psi = synth.random_spinor(DIMS, Ls, seed=45)
    # subnormal inputs are stored with fewer bits: the reference takes what is stored
    psi = np.ldexp(psi.real, log2_psi) + 1j * np.ldexp(psi.imag, log2_psi)
    ref = oracle_lib.dhop(DIMS, Ls, BC, U, psi)
    scale = 2.0 ** -(log2_psi + log2_u) if log2_psi > -1000 else 2.0 ** 1000
    d = (apply(dwf, U, psi, Ls, False) - ref) * scale
    tiny = 2.0 ** -1074 * scale * 100 if log2_psi <= -1000 else 0  # a subnormal's spacing, ~100 roundings
    assert np.all(np.abs(d) <= BOUND * np.abs(psi * scale).max() * 2.0 ** log2_u + tiny)


@pytest.mark.parametrize("c12", [False, True])
def test_non_finite_reals_stay_where_ieee_arithmetic_puts_them(dwf, c12):
    Ls = 6
    U = synth.random_gauge(DIMS, seed=46)
    psi = synth.random_spinor(DIMS, Ls, seed=47)
    clean = apply(dwf, U, psi, Ls, False, c12)
    # [t, z, y, x, s, spin, colour] of the two values
    where = [((1, 0, 2, 1), 3, 0, 1, np.inf), ((3, 1, 5, 0), 2, 3, 2, np.nan)]
    bad = np.zeros(psi.shape, dtype=bool)
    for site, s, spin, colour, value in where:
        psi[site + (s, spin, colour)] = value
        # a hop adds spins in pairs before the link mixes their colours: (0, 3), (1, 2) in x and y,
        # (0, 2), (1, 3) in z and t; both spins of the pair take the product
        for axis in range(4):  # t, z, y, x
            pair = [p for p in (((0, 2), (1, 3)) if axis < 2 else ((0, 3), (1, 2))) if spin in p][0]
            for step in (1, -1):
                n = list(site)
                n[axis] = (n[axis] + step) % psi.shape[axis]
                bad[tuple(n) + (s, list(pair))] = True
    out = apply(dwf, U, psi, Ls, False, c12)
    assert np.array_equal(~np.isfinite(out), bad)
    far = ~bad.any(axis=(-2, -1))  # (site, slice) pairs that do not see the two values
    assert np.array_equal(out[far], clean[far])


def test_zero_field(dwf):
    U = synth.random_gauge(DIMS, seed=48)
    out = apply(dwf, U, np.zeros(DIMS[::-1] + (5, 4, 3), dtype=np.complex128), 5, False)
    assert np.all(out == 0)


def hop_terms(U, psi, dag):
    """Sum of the magnitudes of the terms of every complex component of the hop: over the eight hops of
    a site, sum_b |U_ab| |h_b| with h the projected neighbour (its lower spins repeat the upper ones)."""
    sign = 1 if dag else -1  # forward projector (1 + sign gamma), backward (1 - sign gamma)
    total = np.zeros(psi.shape)
    partner = {0: (3, 2), 1: (3, 2), 2: (2, 3), 3: (2, 3)}
    coeff = {0: (-1j, -1j), 1: (-1, 1), 2: (-1j, 1j), 3: (1, 1)}  # h_k = psi_k + s coeff psi_partner, k = 0, 1
    for mu in range(4):
        axis = 3 - mu
        for back in (0, 1):
            nb = np.roll(psi, 1 if back else -1, axis)
            link = U[..., mu, :, :]
            link = np.roll(link, 1, axis).swapaxes(-1, -2) if back else link
            s = -sign if back else sign
            for k in (0, 1):
                h = nb[..., k, :] + s * coeff[mu][k] * nb[..., partner[mu][k], :]
                t = np.einsum("tzyxab,tzyxsb->tzyxsa", np.abs(link), np.abs(h))
                total[..., k, :] += t
                total[..., partner[mu][k], :] += t
    return total


def graded(kind, psi, U):
    """Fields whose components differ in size by more than a block of integers with one exponent holds, on
    links that leave some of the small ones apart."""
    psi, U = psi.copy(), U.copy()
    if kind == "colours":
        psi *= np.exp2([0, -20, -40])
        U[...] = np.eye(3)
    elif kind == "spins":  # spin 1 takes no part in spin 0's hops
        psi *= np.exp2([-30, 0, -30, -30])[:, None]
    elif kind == "colours and zeros":
        psi *= np.array([1, 0, 2.0 ** -70])
        U[...] = np.eye(3)
    elif kind == "links":
        U[...] = np.diag(np.exp2([0, -25, -50]))
    elif kind == "links and a little mixing":
        U[...] = np.eye(3) + 2.0 ** -58 * U
        psi *= np.array([1, 0, 0])
    elif kind == "one spin":
        psi *= np.array([0, 0, 1, 0])[:, None]
    return psi, U


@pytest.mark.parametrize("kind", ["equal", "colours", "spins", "colours and zeros", "links",
                                  "links and a little mixing", "one spin"])
@pytest.mark.parametrize("Ls", [3, 8])
def test_small_components_beside_large_ones(dwf, oracle_lib, kind, Ls):
    """Every complex component to a precision relative to its own terms. Oracle: at most 24 roundings of a
    term, 24 x 2^-53. Block integers: a hop's truncations and its rounding add up to 11 units of the
    accumulator per real, with the accumulator's own shifts 92 for eight hops, sqrt(2) x 92 for the modulus,
    and they are used only where the |re| + |im| of the hops sum to 2^50 units or more, the moduli of the
    terms to 2^49.5: 1450 x 2^-53. Together 1500 x 2^-53 of the sum of magnitudes."""
    psi, U = graded(kind, synth.random_spinor(DIMS, Ls, seed=51), synth.random_gauge(DIMS, seed=52))
    for dag in (False, True):
        ref = oracle_lib.dhop(DIMS, Ls, BC, U, psi, dag=dag)
        err = np.abs(apply(dwf, U, psi, Ls, dag) - ref)
        assert np.all(err <= 1500 * 2.0 ** -53 * hop_terms(U, psi, dag))


@pytest.mark.parametrize("Ls", [1, 2, 6, 16])
def test_force_of_small_colours_beside_large_ones(dwf, oracle_lib, Ls):
    """Unit links keep the colours apart: entry (a, b) of the gradient is a sum of products of psi's and
    chi's colours a and b, of any size beside the others. 1e-12 as for whole FP64 fields elsewhere."""
    size = np.exp2([0, -20, -40])
    U = synth.unit_gauge(DIMS)
    psi = synth.random_spinor(DIMS, Ls, seed=53) * size
    op = dwf.GridDWF(DIMS, Ls, M5, MASS, bc=BC)
    op.set_gauge(torch.from_numpy(U).cuda())
    _, _, G = op.force(op.pack(torch.from_numpy(psi).cuda(), 0, dwf.FULL))
    _, _, ref = oracle_lib.force(DIMS, Ls, M5, MASS, BC, U, psi)
    s = size[:, None] * size
    assert np.all(np.abs(G.cpu().numpy() - ref) / s <= 1e-12 * np.abs(ref / s).max())
    op.close()

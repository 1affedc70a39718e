"""Every fifth-dimension extent around the limits of the kernels' dispatch, on lattices that full
CTAs do not divide (the launches then take a divisor, or the caller's count and a second launch for the
end), against the FP64 oracle: hopping term and Schur operator (even Ls to 24 and 32 are
compiled in, the rest is generic), the fifth-dimension term (warp shuffles to 32 slice pairs, shared
memory above and for the FP64 inverse), the force (3 to 16 pairs in registers; FP64 in block integers),
and the integer precision conversions bit for bit.

Tolerances as in test_gpu_parity: FP64 1e-12, FP32 1e-5 (force 2e-5), 16-bit storage one output
rounding per launch (2^-11, 2^-8) with the margin used there.
"""
import ctypes

import numpy as np
import pytest
import torch

from paper_2203_06777_gb300 import synth

from .test_gpu_guards import Guarded

pytestmark = pytest.mark.gpu

BC = (1, 1, 1, -1)
M5, MASS = 1.8, 0.01
TOL = {0: 1e-12, 1: 1e-5, 2: 2e-3, 3: 1.6e-2}
TORCH = {1: torch.float32, 2: torch.float16, 3: torch.bfloat16}


@pytest.fixture(scope="module")
def dwf():
    from paper_2203_06777_gb300 import dwf as mod

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    mod.load()
    return mod


def rel(a, b):
    d = np.abs(a - b)
    return float(max(np.linalg.norm(d) / np.linalg.norm(b), d.max() / np.abs(b).max()))


def round_to(x, prec):
    """x rounded once to the storage precision, as float64."""
    if prec == 0:
        return x
    if np.iscomplexobj(x):
        return round_to(x.real, prec) + 1j * round_to(x.imag, prec)
    if prec == 1:
        return x.astype(np.float32).astype(np.float64)
    if prec == 2:
        return x.astype(np.float16).astype(np.float64)
    e = np.maximum(np.frexp(x)[1] - 8, -133)
    return np.ldexp(np.rint(np.ldexp(x, -e)), e)


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("dims,Ls", [((6, 2, 2, 6), 4), ((2, 6, 2, 6), 6), ((6, 6, 2, 2), 7), ((2, 2, 6, 6), 10),
                                     ((6, 2, 6, 2), 11), ((10, 2, 2, 2), 14), ((6, 6, 6, 2), 18), ((2, 6, 6, 2), 20),
                                     ((6, 2, 2, 2), 22), ((2, 2, 2, 6), 24), ((2, 2, 4, 2), 26), ((2, 6, 2, 2), 32),
                                     ((6, 10, 6, 6), 12)])
@pytest.mark.parametrize("prec", [0, 1, 2, 3])
def test_hop_and_schur_operator(dwf, oracle_lib, dims, Ls, prec):
    U = synth.random_gauge(dims, seed=701)
    psi = synth.random_spinor(dims, Ls, seed=702)
    for c12 in (False, True):
        op = dwf.GridDWF(dims, Ls, M5, MASS, bc=BC, compress12=c12)
        op.set_gauge(dev(U))
        U_r = round_to(U, prec)
        if c12:  # the third row is rebuilt from the stored two
            U_r[..., 2, :] = np.cross(U_r[..., 0, :], U_r[..., 1, :]).conj()
        psi_r = round_to(psi, prec)
        out = op.unpack(op.dhop(op.pack(dev(psi), prec, dwf.FULL), dwf.FULL)).cpu().numpy()
        assert rel(out, oracle_lib.dhop(dims, Ls, BC, U_r, psi_r)) < TOL[prec]
        odd = oracle_lib.parity_mask(dims)[..., None, None, None]
        f = op.pack(dev(psi), prec, dwf.ODD)
        for dag in (False, True):
            got = op.unpack(op.mpc(f, dag=dag), subset=dwf.ODD).cpu().numpy()
            if dag:
                want = psi_r * odd  # Mpc^+ from its definition by the oracle's pieces
                te = oracle_lib.mooee(dims, Ls, M5, MASS, oracle_lib.dhop(dims, Ls, BC, U_r, want, dag=True) * ~odd,
                                      dag=True, inverse=True)
                want = oracle_lib.mooee(dims, Ls, M5, MASS, want, dag=True) - 0.25 * odd * oracle_lib.dhop(
                    dims, Ls, BC, U_r, te, dag=True)
            else:
                want = oracle_lib.mpc(dims, Ls, M5, MASS, BC, U_r, psi_r * odd)
            assert rel(got * odd, want * odd) < TOL[prec] * (4 if prec > 1 else 1), (c12, dag)
        op.close()


@pytest.mark.parametrize("Ls", [1, 2, 3, 4, 5, 9, 16, 17, 31, 32, 33, 62, 63, 64, 65, 66, 128])
@pytest.mark.parametrize("prec", [0, 1, 2, 3])
def test_fifth_dimension_term(dwf, oracle_lib, Ls, prec):
    dims = (2, 2, 4, 2)
    op = dwf.GridDWF(dims, Ls, M5, MASS)
    psi = synth.random_spinor(dims, Ls, seed=711)
    f = op.pack(dev(psi), prec, dwf.FULL)
    psi_r = round_to(psi, prec)
    for dag in (False, True):
        for inverse in (False, True):
            ref = oracle_lib.mooee(dims, Ls, M5, MASS, psi_r, dag=dag, inverse=inverse)
            out = op.mooee(f, dag=dag, inverse=inverse)
            assert rel(op.unpack(out).cpu().numpy(), ref) < TOL[prec], (dag, inverse)
            g = f.clone()
            assert torch.equal(op.mooee(g, dag=dag, inverse=inverse, out=g), out)  # in place
    op.close()


@pytest.mark.parametrize("Ls", [1, 2, 5, 6, 7, 8, 9, 13, 16, 18, 23, 31, 33])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("c12", [False, True])
def test_force(dwf, oracle_lib, Ls, prec, c12):
    dims = (4, 2, 6, 2)
    U = synth.random_gauge(dims, seed=721)
    psi = synth.random_spinor(dims, Ls, seed=722)
    op = dwf.GridDWF(dims, Ls, M5, MASS, bc=BC, compress12=c12)
    op.set_gauge(dev(U))
    f = op.pack(dev(psi), prec, dwf.FULL)
    U_r = round_to(U, prec)
    if c12:
        U_r[..., 2, :] = np.cross(U_r[..., 0, :], U_r[..., 1, :]).conj()
    S, F, G = op.force(f)
    S_ref, F_ref, G_ref = oracle_lib.force(dims, Ls, M5, MASS, BC, U_r, round_to(psi, prec))
    tol = 1e-12 if prec == 0 else 2e-5
    assert abs(S - S_ref) < tol * S_ref
    assert rel(F.cpu().numpy(), F_ref) < tol and rel(G.cpu().numpy(), G_ref) < tol
    F2, G2 = op.force_contract(f, op.m(f))  # the contraction alone
    assert torch.equal(F2, F) and torch.equal(G2, G)
    op.close()


@pytest.mark.parametrize("log2,spread", [(0, 20), (-420, 0), (420, 0), (-150, 30)])
def test_force_fp64_magnitudes(dwf, oracle_lib, log2, spread):
    """Slices of very different magnitude, and fields outside the integer range (IEEE products)."""
    dims, Ls = (4, 2, 2, 4), 6
    U = synth.random_gauge(dims, seed=731)
    psi = synth.random_spinor(dims, Ls, seed=732)
    psi *= np.exp2(np.random.default_rng(733).integers(-spread, spread + 1, Ls))[:, None, None]
    op = dwf.GridDWF(dims, Ls, M5, MASS, bc=BC)
    op.set_gauge(dev(U))
    _, F, G = op.force(op.pack(dev(psi * 2.0 ** log2), 0, dwf.FULL))
    _, F_ref, G_ref = oracle_lib.force(dims, Ls, M5, MASS, BC, U, psi)
    s = 2.0 ** -log2  # F and G are quadratic in psi
    assert rel(F.cpu().numpy() * s * s, F_ref) < 1e-12 and rel(G.cpu().numpy() * s * s, G_ref) < 1e-12
    op.close()


def values(kind, n):
    rng = np.random.default_rng(741)
    if kind == "bits":  # every exponent, subnormals, infinities and NaN among them
        return rng.integers(-(2 ** 63), 2 ** 63, n, dtype=np.int64).view(np.float64)
    x = rng.normal(size=n)
    if kind == "ties":  # halfway between neighbouring FP32 values, and just off
        x = x.astype(np.float32).astype(np.float64) * (1 + 2.0 ** -24)
        x[::2] = np.nextafter(x[::2], np.inf)
        return x
    x *= np.exp(12 * rng.normal(size=n))
    x[:8] = [0.0, -0.0, np.inf, np.nan, 1e39, 3.4028235677973366e38, 65519.99, 65520.0]
    return x


@pytest.mark.parametrize("kind", ["bits", "wide", "ties"])
@pytest.mark.parametrize("scale", [1.0, 0.75, -3.3e-5, 1e-310, 7.1e30, 0.0])
def test_conversions_round_once(dwf, kind, scale):
    dims, Ls = (4, 4, 4, 2), 7
    op = dwf.GridDWF(dims, Ls, M5, MASS)
    rv = {0: 1, 1: 2, 2: 4, 3: 4}

    def by_real(t, prec):  # flat layout -> one order of the values for every precision
        return t.reshape(-1, 24 // rv[prec], 4, (Ls + 1) // 2, rv[prec], 2).permute(0, 2, 3, 5, 1, 4).reshape(-1)

    f = dev(values(kind, 2 * op.half_reals))
    with np.errstate(all="ignore"):
        exact = by_real(f, 0).cpu().numpy() * scale
        for prec in (1, 2):
            out = by_real(op.convert(f, prec, scale=scale), prec).cpu().numpy()
            assert np.array_equal(out, exact.astype(out.dtype), equal_nan=True), prec
        out = by_real(op.convert(f, 3, scale=scale).double(), 3).cpu().numpy()
        finite = np.abs(exact) < 3.38e38  # (the reference below knows no overflow)
        assert np.array_equal(out[finite], round_to(exact[finite], 3))
        for prec in (1, 2, 3):
            low = f.to(TORCH[prec])
            out = by_real(op.convert(low, 0, scale=scale), 0).cpu().numpy()
            assert np.array_equal(out, by_real(low, prec).double().cpu().numpy() * scale, equal_nan=True), prec
    op.close()


@pytest.mark.parametrize("scale", [1e300, -1e280, 2.0 ** 897, 2.0 ** 896, 1e-290, -1e-300, 2.0 ** -899, 2.0 ** -898])
def test_conversions_at_extreme_scales(dwf, scale):
    """Zeros, subnormals, infinities and NaN times a scale whose exponent alone would bring them into the
    range of normal FP32 numbers; and normal values that the scale brings there."""
    dims, Ls = (4, 2, 2, 2), 3
    op = dwf.GridDWF(dims, Ls, M5, MASS)
    n = 2 * op.half_reals
    special = [0.0, -0.0, 5e-324, -1e-310, 2.2e-308, np.inf, -np.inf, np.nan, 1.7e308]
    x = np.resize(np.concatenate([special, values("bits", 501), np.random.default_rng(742).normal(size=64) / scale]), n)
    # the same values at the same places of the field for every precision: one value per (site, slice)
    psi = np.broadcast_to(x[:op.half_reals // 12].reshape(dims[::-1] + (Ls + 1, 1, 1))[..., :Ls, :, :],
                          op.canonical_shape()).astype(np.complex128)
    f = op.pack(dev(psi), 0, dwf.FULL)
    with np.errstate(all="ignore"):
        exact = x[:op.half_reals // 12].reshape(dims[::-1] + (Ls + 1,))[..., :Ls] * scale
        for prec in (1, 2, 3):
            low = op.convert(f, prec, scale=scale)
            out = op.unpack(low).cpu().numpy().real
            want = exact.astype(np.float32 if prec == 1 else np.float16) if prec < 3 else exact
            if prec == 3:
                finite = np.abs(exact) < 3.38e38
                assert np.array_equal(out[finite][:, 0, 0], round_to(exact[finite], 3))
                assert np.array_equal(np.isnan(out[..., 0, 0]), np.isnan(exact))
            else:
                assert np.array_equal(out[..., 0, 0], want.astype(np.float64), equal_nan=True), prec
            rv = {1: 2, 2: 4, 3: 4}[prec]
            assert not low.reshape(-1, 24 // rv, 4, (Ls + 1) // 2, rv, 2)[:, :, :, -1, :, 1].any()  # the pad slice
    op.close()


@pytest.mark.parametrize("Ls", [2, 3, 8, 11, 12, 16, 24, 64])
@pytest.mark.parametrize("prec", [0, 1, 2, 3])
def test_fifth_dimension_inverse_keeps_non_finite_values_on_their_line(dwf, Ls, prec):
    """The inverse couples the slices of one real of one site: nothing else may see an infinity or NaN."""
    dims = (4, 2, 6, 4)
    psi = synth.random_spinor(dims, Ls, seed=751)
    op = dwf.GridDWF(dims, Ls, M5, MASS)
    rng = np.random.default_rng(752)
    where = rng.random(dims[::-1] + (4, 3)) < 0.02  # [t, z, y, x, spin, colour]
    bad = psi.copy()
    for idx in np.argwhere(where):
        s = rng.integers(Ls)
        bad[tuple(idx[:4]) + (s,) + tuple(idx[4:])] = complex([np.inf, -np.inf, np.nan][rng.integers(3)], 0.5)
    line = np.broadcast_to(where[:, :, :, :, None], psi.shape)  # only real parts are planted
    for dag in (False, True):
        clean = op.unpack(op.mooee(op.pack(dev(psi), prec, dwf.FULL), dag=dag, inverse=True)).cpu().numpy()
        out = op.unpack(op.mooee(op.pack(dev(bad), prec, dwf.FULL), dag=dag, inverse=True)).cpu().numpy()
        assert np.array_equal(~np.isfinite(out.real), line)
        assert np.array_equal(out.real[~line], clean.real[~line])
        assert np.isfinite(out.imag).all() and np.array_equal(out.imag[~line], clean.imag[~line])
    op.close()


def test_fifth_dimension_term_of_more_than_2_32_vectors(dwf):
    """A field with more 16-byte vectors per slice pair than 32 bits count (77 GB, in place): every site of a
    constant field has the value of the first."""
    dims, Ls = (128, 128, 128, 96), 2
    nbytes = int(np.prod(dims)) * Ls * 24 * 8
    assert int(np.prod(dims)) * 24 > 2 ** 32
    if torch.cuda.mem_get_info()[0] < nbytes + 2 ** 33:
        pytest.skip("needs 86 GB of free device memory")
    small = dwf.GridDWF((2, 2, 2, 2), Ls, M5, MASS)
    want = small.mooee(torch.ones(2 * small.half_reals, dtype=torch.float64, device="cuda"))[:4 * Ls * 24]
    op = dwf.GridDWF(dims, Ls, M5, MASS)
    f = torch.ones(2 * op.half_reals, dtype=torch.float64, device="cuda")
    op.mooee(f, out=f)
    for part in f.view(-1, 4 * Ls * 24).split(2 ** 22):
        assert bool((part == want).all())
    small.close()
    op.close()
    del f, part
    torch.cuda.empty_cache()


@pytest.mark.parametrize("dims,Ls,spc", [((6, 2, 2, 6), 10, None), ((6, 10, 6, 6), 12, None), ((6, 10, 6, 6), 12, 7),
                                         ((2, 6, 2, 6), 7, 5), ((6, 10, 6, 22), 6, 7)])
def test_ragged_ends_and_short_warps(dwf, oracle_lib, monkeypatch, dims, Ls, spc):
    """CTAs whose last warp is short (120 threads in the first two cases), and sites per CTA that do not
    divide the half lattice, so that its end takes a launch of its own (the last case with more than
    512 partial sums in either kind of reducing launch). Sums: 48 squares per thread in FP32, all of one
    sign, 48 x 2^-24."""
    U, psi = synth.random_gauge(dims, seed=761, eps=0.3), synth.random_spinor(dims, Ls, seed=762)
    plain = dwf.GridDWF(dims, Ls, M5, MASS, bc=BC)
    if spc:
        monkeypatch.setenv("GRID_DWF_SITES_PER_CTA", str(spc))
    op = dwf.GridDWF(dims, Ls, M5, MASS, bc=BC)
    for o in (plain, op):
        o.set_gauge(dev(U))
    half = op.half_reals
    for prec in (1, 2, 3):
        f = op.pack(dev(psi), prec, dwf.FULL)
        calls = {"dhop": lambda o, out: o.dhop(f, dwf.FULL, out=out), "m": lambda o, out: o.m(f, dag=True, out=out),
                 "mpc": lambda o, out: o.mpc(f[half:].clone(), out=out),
                 "mdagm": lambda o, out: o.mdagm(f[half:].clone(), out=out)}
        for name, call in calls.items():
            g = Guarded(f.numel() if name in ("dhop", "m") else half, f.dtype)
            call(op, g.t)
            g.check(name)
            assert torch.equal(g.t, call(plain, None)), name
    f = op.pack(dev(psi), 1, dwf.FULL)
    for _ in range(3):
        S, _, _ = op.force(f, want_F=False, want_G=False)
        assert abs(S - op.norm2(op.m(f))) < 48 * 2.0 ** -24 * S
    b = op.pack(dev(psi), 0, dwf.FULL)
    _, ref = plain.cg(b, tol=1e-10, maxiter=5000, mode=dwf.CG_FP64)
    for mode in (1, 2, 3):
        x, st = op.cg(b, tol=1e-10, maxiter=5000, mode=mode)
        assert st.converged and st.iterations < (1.2 if mode == 1 else 2) * ref.iterations
        r = oracle_lib.m(dims, Ls, M5, MASS, BC, U, op.unpack(x).cpu().numpy()) - psi
        assert np.linalg.norm(r) < 1e-8 * np.linalg.norm(psi)
    plain.close()
    op.close()


@pytest.mark.parametrize("Ls", [5, 8, 12, 18, 34])
@pytest.mark.parametrize("prec", [0, 1])
def test_force_outputs_between_16_byte_boundaries(dwf, Ls, prec):
    """F and G at odd multiples of 8 bytes: the same numbers, to FP32 rounding of a sum in another order."""
    dims = (4, 2, 2, 4)
    op = dwf.GridDWF(dims, Ls, M5, MASS, bc=BC)
    op.set_gauge(dev(synth.random_gauge(dims, seed=781)))
    f = op.pack(dev(synth.random_spinor(dims, Ls, seed=782)), prec, dwf.FULL)
    chi = op.m(f)
    _, F, G = op.force(f)
    out = torch.zeros(2, F.numel() * 2 + 2, dtype=torch.float64, device="cuda")
    at = [ctypes.c_void_p(row.data_ptr() + 8) for row in out]
    op._call("grid_dwf_force_contract", prec, dwf._ptr(f), dwf._ptr(chi), *at)
    for row, want in zip(out.cpu().numpy(), (F, G)):
        assert row[0] == 0 and row[-1] == 0
        got = row[1:-1].view(np.complex128).reshape(want.shape)
        assert rel(got, want.cpu().numpy()) < (1e-14 if prec == 0 else 2e-5)
    op.close()

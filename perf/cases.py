"""The work that programs using the domain-wall operator library have it do, as measured cases.

A case names one call (or one short sequence that belongs together) of the public binding
``paper_2203_06777_gb300.dwf`` with a lattice (Lx, Ly, Lz, Lt), a fifth-dimension extent Ls, a
storage precision and the options of that call. The kinds:

  dhop    the hopping term (DhopEO, DhopOE or both halves), the operator's kernel
  mpc     the Schur complement Mpc or its adjoint on the odd half field
  mdagm   Mpc^+ Mpc, what a CG iteration or a true residual applies
  mooee   the fifth-dimension term or its inverse on its own
  layout  canonical field -> device layout -> canonical field (input and output of a program)
  blas    precision conversion, norm and inner product, the vector steps of a caller's own solver
  force   |M psi|^2 with its su(3) force and ambient gradient
  action  the same action through autograd: value, dS/dpsi and dS/dU (forward and backward)
  cg      M x = b to 1e-10 through the Schur system, plain or mixed precision

Links are random SU(3) matrices near the identity (disorder of the size of the library's own
workloads), fields are complex Gaussian, M5 = 1.8, m = 0.01, antiperiodic in t. Lattices and
extents are those of the repository's workloads and parity tests (4^4 x 8, 16^4 x 16, 24^4 x 12,
32^4 x 16, ragged boxes with odd Ls).
"""
import math

import torch

from paper_2203_06777_gb300 import dwf

M5, MASS = 1.8, 0.01
BC = (1, 1, 1, -1)
PREC = {"fp64": dwf.FP64, "fp32": dwf.FP32, "fp16": dwf.FP16, "bf16": dwf.BF16}
DTYPE = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}
BYTES = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}
MODE = {"fp64": dwf.CG_FP64, "fp32": dwf.CG_MIXED_FP32, "fp16": dwf.CG_MIXED_FP16, "bf16": dwf.CG_MIXED_BF16}
PARITY = {"even": dwf.EVEN, "odd": dwf.ODD, "full": dwf.FULL}


def _case(kind, lx, ly, lz, lt, ls, prec, parity="full", dag=False, inverse=False, c12=False):
    return {"kind": kind, "lx": lx, "ly": ly, "lz": lz, "lt": lt, "ls": ls, "prec": prec, "parity": parity,
            "dag": dag, "inverse": inverse, "c12": c12}


def listed():
    cases = {
        # a test lattice or the coarsest level of a tuning run: launch and call latency
        "dhop_4x4x4x4_ls8_fp32": _case("dhop", 4, 4, 4, 4, 8, "fp32"),
        # the benchmark workload
        "dhop_16x16x16x16_ls16_fp32": _case("dhop", 16, 16, 16, 16, 16, "fp32"),
        # the largest lattice of the library's workloads, storage of a 16-bit inner solver
        "dhop_32x32x32x32_ls16_bf16": _case("dhop", 32, 32, 32, 32, 16, "bf16"),
        # adjoint Schur operator of the FP16 inner solver at production size
        "mpc_dag_24x24x24x24_ls12_fp16": _case("mpc", 24, 24, 24, 24, 12, "fp16", "odd", dag=True),
        # a box with unequal sides, an extent with no compiled specialisation and 12-real links
        "mdagm_14x10x6x18_ls10_fp32_c12": _case("mdagm", 14, 10, 6, 18, 10, "fp32", "odd", c12=True),
        # the FP64 operator behind every true residual and the plain FP64 solver
        "mdagm_16x16x16x16_ls16_fp64": _case("mdagm", 16, 16, 16, 16, 16, "fp64", "odd"),
        # the preconditioner step of a caller's own solver
        "mooee_inv_24x24x24x24_ls12_fp32": _case("mooee", 24, 24, 24, 24, 12, "fp32", inverse=True),
        # a field handed to the library and taken back
        "layout_16x16x16x16_ls16_fp32": _case("layout", 16, 16, 16, 16, 16, "fp32"),
        # conversion to the inner precision, |a|^2 and (a, b)
        "blas_24x24x24x24_ls12_fp32": _case("blas", 24, 24, 24, 24, 12, "fp32", "odd"),
        # the force of a molecular-dynamics step, FP32 fields
        "force_16x16x16x16_ls16_fp32": _case("force", 16, 16, 16, 16, 16, "fp32"),
        # a gradient step through autograd at the default (FP64) precision
        "action_8x8x8x8_ls8_fp64": _case("action", 8, 8, 8, 8, 8, "fp64"),
        # the solve that production runs spend their time in
        "cg_mixed_16x16x16x16_ls12_fp32": _case("cg", 16, 16, 16, 16, 12, "fp32"),
    }
    return [dict(c, name=n) for n, c in cases.items()]


# (weight, precisions, smallest and largest number of 5D sites) of each kind. The largest listed case
# applies the 16-bit hop to 16.8 M five-dimensional sites; the ranges of the dearer kinds end where
# a pass costs about as much at the start.
RANGES = {
    "dhop": (5, ("fp64", "fp32", "fp16", "bf16"), 1 << 11, 1 << 23),
    "mpc": (3, ("fp64", "fp32", "fp16", "bf16"), 1 << 11, 1 << 22),
    "mdagm": (3, ("fp64", "fp32", "fp16", "bf16"), 1 << 11, 1 << 22),
    "mooee": (1, ("fp64", "fp32", "fp16", "bf16"), 1 << 11, 1 << 22),
    "layout": (1, ("fp64", "fp32", "fp16", "bf16"), 1 << 11, 1 << 21),
    "blas": (1, ("fp32", "fp16", "bf16"), 1 << 11, 1 << 22),
    "force": (2, ("fp64", "fp32"), 1 << 11, 1 << 20),
    "action": (1, ("fp64", "fp32"), 1 << 11, 1 << 18),
    "cg": (1, ("fp64", "fp32", "fp16", "bf16"), 1 << 11, 1 << 16),
}


def draw(rng):
    kind = rng.choices(list(RANGES), [r[0] for r in RANGES.values()])[0]
    _, precs, lo, hi = RANGES[kind]
    while True:
        ls = rng.choice((rng.randint(4, 24), 8, 10, 12, 16, 16, 24))
        n5 = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        side = (n5 / ls) ** 0.25
        dims = [max(2, 2 * round(side * math.exp(rng.uniform(-0.5, 0.5)) / 2)) for _ in range(4)]
        if max(dims) <= 48 and lo // 2 <= math.prod(dims) * ls <= hi:
            break
    prec = rng.choice(precs)
    parity = "full" if kind in ("force", "action", "layout", "cg") else "odd"
    if kind in ("dhop", "mooee", "blas"):
        parity = rng.choice(("even", "odd", "full"))
    return _case(kind, *dims, ls, prec, parity, dag=kind in ("dhop", "mpc", "mooee") and rng.random() < 0.5,
                 inverse=kind == "mooee" and rng.random() < 0.5, c12=rng.random() < 0.2)


# ---------------------------------------------------------------- inputs


def _dims(case):
    return case["lx"], case["ly"], case["lz"], case["lt"]


def _shape4(case):
    return case["lt"], case["lz"], case["ly"], case["lx"]


def _complex_gaussian(shape, seed, device):
    g = torch.Generator(device=device)
    g.manual_seed(seed)
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), generator=g, device=device,
                                             dtype=torch.float64) * math.sqrt(0.5))


def _links(case, seed, device):
    """SU(3) matrices near the identity: 1 + 0.4 i (complex Gaussian), rows made orthonormal."""
    a = 0.4j * _complex_gaussian(_shape4(case) + (4, 2, 3), 2 * seed + 1, device)
    a[..., 0, 0] += 1
    a[..., 1, 1] += 1
    r0, r1 = a[..., 0, :], a[..., 1, :]
    r0 = r0 / r0.abs().square().sum(-1, keepdim=True).sqrt()
    r1 = r1 - (r0.conj() * r1).sum(-1, keepdim=True) * r0
    r1 = r1 / r1.abs().square().sum(-1, keepdim=True).sqrt()
    r2 = torch.linalg.cross(r0, r1).conj()
    return torch.stack((r0, r1, r2), -2).contiguous()


def _spinor(case, seed, device):
    return _complex_gaussian(_shape4(case) + (case["ls"], 4, 3), 2 * seed, device)


def _second(case, psi, seed):
    """A field with an overlap of order one with psi, as successive vectors of a solver have."""
    return (0.8 + 0.6j) * psi + 0.3 * _spinor(case, seed + 7919, psi.device)


def _subset(case):
    """Subset of the input field: DhopEO (output even) reads the odd half and the other way round."""
    if case["parity"] == "full":
        return dwf.FULL
    if case["kind"] == "dhop":
        return dwf.ODD if case["parity"] == "even" else dwf.EVEN
    return PARITY[case["parity"]]


def prepare(case, seed):
    device = torch.device("cuda", torch.cuda.current_device())
    kind, prec = case["kind"], PREC[case["prec"]]
    op = dwf.GridDWF(_dims(case), case["ls"], M5, MASS, bc=BC, compress12=case["c12"])
    U = _links(case, seed, device)
    psi = _spinor(case, seed, device)
    st = {"case": case, "op": op}
    if kind == "action":
        st["U"], st["psi"] = U.requires_grad_(), psi.requires_grad_()
        return st
    if kind not in ("mooee", "layout", "blas"):
        op.set_gauge(U)
    if kind == "layout":
        st["psi"] = psi
        st["field"] = op.field(prec, dwf.FULL)
        st["back"] = torch.empty_like(psi)
    elif kind == "blas":
        st["f64"] = op.pack(psi, dwf.FP64, _subset(case))
        st["b"] = op.pack(_second(case, psi, seed), prec, _subset(case))
        st["a"] = torch.empty_like(st["b"])
    elif kind == "cg":
        st["b"] = op.pack(psi, dwf.FP64, dwf.FULL)
    else:
        st["f"] = op.pack(psi, prec, _subset(case))
        if kind != "force":
            st["out"] = torch.empty_like(st["f"])
    return st


SCALE = 0.75  # of the blas case's conversion


def run(state):
    case, op = state["case"], state["op"]
    kind, prec = case["kind"], PREC[case["prec"]]
    if kind == "dhop":
        return op.dhop(state["f"], PARITY[case["parity"]], dag=case["dag"], out=state["out"])
    if kind == "mpc":
        return op.mpc(state["f"], dag=case["dag"], out=state["out"])
    if kind == "mdagm":
        return op.mdagm(state["f"], out=state["out"])
    if kind == "mooee":
        return op.mooee(state["f"], dag=case["dag"], inverse=case["inverse"], out=state["out"])
    if kind == "layout":
        f = op.pack(state["psi"], prec, dwf.FULL, out=state["field"])
        return f, op.unpack(f, out=state["back"])
    if kind == "blas":
        a = op.convert(state["f64"], prec, SCALE, out=state["a"])
        z = op.inner(a, state["b"])
        return a, op.norm2(a), z.real, z.imag
    if kind == "force":
        return op.force(state["f"])
    if kind == "action":
        s = dwf.dwf_action(state["psi"], state["U"], op, prec)
        g_psi, g_u = torch.autograd.grad(s, (state["psi"], state["U"]))
        return s.detach(), g_psi, g_u
    return op.cg(state["b"], tol=1e-10, mode=MODE[case["prec"]])[0]


# ---------------------------------------------------------------- cost

HOP_FLOPS = 1320  # per 5D output site of one half-lattice hop


def work(case):
    v = math.prod(_dims(case))
    n5 = v * case["ls"]
    b = BYTES[case["prec"]]
    half = n5 // 2 * 24 * b
    links = v * 4 * (12 if case["c12"] else 18) * b
    kind = case["kind"]
    sub = 2 if case["parity"] == "full" else 1
    if kind == "dhop":
        return {"bytes": 2 * sub * half + links, "flops": HOP_FLOPS * n5 // 2 * sub}
    if kind in ("mpc", "mdagm"):
        # input once, output once; every link once
        hops = 2 if kind == "mpc" else 4
        return {"bytes": 2 * half + links, "flops": hops * (HOP_FLOPS + 96) * n5 // 2}
    if kind == "mooee":
        return {"bytes": 2 * sub * half, "flops": (4 if case["inverse"] else 3) * 24 * n5 // 2 * sub}
    if kind == "layout":
        return {"bytes": 2 * (n5 * 24 * 8 + 2 * half), "flops": 0}
    if kind == "blas":
        # FP64 in and converted out; then both operands of the inner product (the norm's is one of them)
        return {"bytes": sub * (n5 // 2 * 24 * 8 + 3 * half), "flops": 7 * 24 * n5 // 2 * sub}
    canon = v * 4 * 18 * 8
    if kind == "force":
        # psi and the links in, F and G out; M psi, eight outer products per site and direction pair
        return {"bytes": 2 * half + links + 2 * canon, "flops": (HOP_FLOPS + 1500) * n5}
    if kind == "action":
        return {"bytes": 2 * (n5 * 24 * 8 + canon), "flops": (2 * HOP_FLOPS + 1500) * n5}
    # cg: links and source in, solution out; about 120 applications of four half hops
    return {"bytes": 2 * n5 * 24 * 8 + v * 4 * 18 * 8, "flops": 120 * 4 * HOP_FLOPS * n5 // 2}


def tolerance(case):
    kind, prec = case["kind"], case["prec"]
    if kind == "layout":
        return "exact"  # one rounding per value, and back
    if kind == "cg":
        # two solutions to a true residual of 1e-10 differ by that times a condition number
        # (seen against the 64-bit solution: 1.4e-9, largest difference 2.1e-8)
        return {"rel": 6e-9, "max": 1e-7}
    if prec == "fp64":
        return {"rel": 1.5e-15, "max": 8e-15}  # seen: 3.5e-16, 1.6e-15
    if prec == "fp32":
        return {"rel": 5e-7, "max": 3e-6}  # seen: 1.3e-7, 6.4e-7
    # one output rounding per launch, unit roundoff 2^-11 (fp16) or 2^-8 (bf16); seen in those units:
    # 0.43 and 1.9 for one launch, 0.45 and 3.4 for mpc, 0.6 and 2.9 for mdagm
    unit = 2.0 ** -11 if prec == "fp16" else 2.0 ** -8
    rel, largest = {"mpc": (2, 14), "mdagm": (2.5, 14)}.get(kind, (2, 8))
    return {"rel": rel * unit, "max": largest * unit}


# ---------------------------------------------------------------- 64-bit reference (plain torch)

_I = 1j
GAMMA = (
    ((0, 0, 0, -_I), (0, 0, -_I, 0), (0, _I, 0, 0), (_I, 0, 0, 0)),
    ((0, 0, 0, -1), (0, 0, 1, 0), (0, 1, 0, 0), (-1, 0, 0, 0)),
    ((0, 0, -_I, 0), (0, 0, 0, _I), (_I, 0, 0, 0), (0, -_I, 0, 0)),
    ((0, 0, 1, 0), (0, 0, 0, 1), (1, 0, 0, 0), (0, 1, 0, 0)),
)


def _shift(x, mu, step):
    """x at the neighbour in direction +mu (step 1) or -mu (step -1), with the boundary phase."""
    dim = 3 - mu
    y = torch.roll(x, -step, dim)
    if BC[mu] < 0:
        edge = y.shape[dim] - 1 if step > 0 else 0
        sign = torch.ones(y.shape[dim], dtype=torch.float64, device=y.device)
        sign[edge] = -1
        y = y * sign.view([-1 if d == dim else 1 for d in range(y.dim())])
    return y


def _hop(U, psi, dag):
    out = 0
    eye = torch.eye(4, dtype=psi.dtype, device=psi.device)
    sgn = 1 if dag else -1
    for mu in range(4):
        gam = torch.tensor(GAMMA[mu], dtype=psi.dtype, device=psi.device)
        u = U[..., mu, :, :].unsqueeze(-3)  # [t, z, y, x, 1, a, b]
        # psi is [t, z, y, x, s, spin, colour]; multiply colour by u, spin by the projector
        fwd = _shift(psi, mu, 1) @ u.transpose(-1, -2)
        bwd = _shift(psi @ u.conj(), mu, -1)
        out = out + (eye + sgn * gam) @ fwd + (eye - sgn * gam) @ bwd
    return out


def _mooee_matrices(ls, dag, inverse, device):
    """The Ls x Ls matrices of the upper and the lower two spins."""
    up = torch.eye(ls, dtype=torch.float64) * (5.0 - M5)
    for s in range(ls):
        up[s, (s - 1) % ls] += -1.0 if s > 0 else MASS
    lo = torch.eye(ls, dtype=torch.float64) * (5.0 - M5)
    for s in range(ls):
        lo[s, (s + 1) % ls] += -1.0 if s < ls - 1 else MASS
    if dag:
        up, lo = up.T, lo.T
    if inverse:
        up, lo = torch.linalg.inv(up), torch.linalg.inv(lo)
    return up.to(device), lo.to(device)


def _mooee(psi, dag, inverse=False):
    ls = psi.shape[4]
    up, lo = (m.to(psi.dtype) for m in _mooee_matrices(ls, dag, inverse, psi.device))
    flat = psi.reshape(psi.shape[:4] + (ls, 12))
    return torch.cat((up @ flat[..., :6], lo @ flat[..., 6:]), -1).reshape(psi.shape)


def _odd_mask(case, device):
    t, z, y, x = (torch.arange(n, device=device) for n in _shape4(case))
    p = (t[:, None, None, None] + z[:, None, None] + y[:, None] + x) % 2
    return (p == 1).to(torch.float64)[..., None, None, None]


def _m(U, psi, dag):
    return _mooee(psi, dag) - 0.5 * _hop(U, psi, dag)


def _mpc(U, psi, dag, odd):
    te = _mooee(_hop(U, psi, dag) * (1 - odd), dag, inverse=True)
    return _mooee(psi, dag) - 0.25 * _hop(U, te, dag) * odd


def _round(x, prec):
    """x rounded once to the storage precision (a torch conversion from 64 to 16 bits rounds twice)."""
    if prec == "fp64":
        return x
    x = torch.view_as_real(x)
    if prec == "fp32":
        return torch.view_as_complex(x.to(torch.float32).to(torch.float64))
    bits, lowest = (11, -24) if prec == "fp16" else (8, -133)
    e = torch.frexp(x)[1].to(torch.int64).sub(bits).clamp_(min=lowest)
    unit = ((e + 1023) << 52).view(torch.float64)  # 2^e, the spacing of the stored values around x
    return torch.view_as_complex(torch.round(x / unit) * unit)


def _stored_links(case, U):
    """The links as the handle holds them in the case's precision."""
    U = _round(U, case["prec"])
    if case["c12"]:
        r0, r1 = U[..., 0, :], U[..., 1, :]
        U = torch.stack((r0, r1, torch.linalg.cross(r0, r1).conj()), -2)
    return U


def _device_layout(case, psi, subset, prec):
    """A canonical field as the flat device layout: per parity, blocks of 4 sites of
    [16-byte chunk][site][slice pair][real][slice]."""
    ls = case["ls"]
    lsp = ls + ls % 2
    lt, lz, ly, lx = _shape4(case)
    rv = 8 // BYTES[prec]
    halves = []
    for par in ((0, 1) if subset == dwf.FULL else (subset,)):
        t, z, y, h = torch.meshgrid(*(torch.arange(n, device=psi.device) for n in (lt, lz, ly, lx // 2)), indexing="ij")
        x = 2 * h + (par + t + z + y) % 2
        f = torch.view_as_real(psi)[t, z, y, x].reshape(-1, ls, 24)
        if lsp != ls:
            f = torch.cat((f, f.new_zeros(f.shape[0], 1, 24)), 1)
        f = f.reshape(-1, 4, lsp // 2, 2, 24 // rv, rv)  # block, site, pair, slice, chunk, real
        halves.append(f.permute(0, 4, 1, 2, 5, 3).reshape(-1))
    return torch.cat(halves)


def exact(case, seed):
    kind, prec, dag = case["kind"], case["prec"], case["dag"]
    device = torch.device("cuda", torch.cuda.current_device())
    psi = _spinor(case, seed, device)
    odd = _odd_mask(case, device)
    if kind == "layout":
        psi = _round(psi, prec)
        return _device_layout(case, psi, dwf.FULL, prec).to(DTYPE[prec]), psi
    if kind == "mooee":
        return _device_layout(case, _mooee(_round(psi, prec), dag, case["inverse"]), _subset(case), prec)
    if kind == "blas":
        sub = _subset(case)
        mask = 1.0 if sub == dwf.FULL else odd if sub == dwf.ODD else 1 - odd
        a = SCALE * psi
        z = (_round(a, prec).conj() * _round(_second(case, psi, seed), prec) * mask).sum()
        n = (_round(a, prec).abs().square() * mask).sum()
        return _device_layout(case, a, sub, prec), n.item(), z.real.item(), z.imag.item()
    U = _links(case, seed, device)
    if kind in ("force", "action"):
        psi = _round(psi, prec).requires_grad_()
        U = _stored_links(case, U).requires_grad_()
        s = _m(U, psi, False).abs().square().sum()
        g_psi, g_u = torch.autograd.grad(s, (psi, U))
        s = s.detach()
        if kind == "action":
            return s, g_psi, g_u
        w = g_u @ U.detach().conj().transpose(-1, -2)
        f = 0.5 * (w - w.conj().transpose(-1, -2))
        tr = torch.diagonal(f, dim1=-2, dim2=-1).sum(-1)[..., None, None]
        return s.item(), f - tr / 3 * torch.eye(3, dtype=f.dtype, device=device), g_u
    if kind == "cg":
        return _exact_solve(case, U, psi, odd)
    U, psi = _stored_links(case, U), _round(psi, prec)
    if kind == "dhop":
        sub = PARITY[case["parity"]]
        return _device_layout(case, _hop(U, psi, dag), sub, prec)
    psi = psi * odd
    out = _mpc(U, psi, dag if kind == "mpc" else False, odd)
    if kind == "mdagm":
        out = _mpc(U, out, True, odd)
    return _device_layout(case, out, dwf.ODD, prec)


def _exact_solve(case, U, b, odd):
    """M x = b by CG on the Schur normal equations, well past the tolerance of the measured call
    (None on lattices where that takes long)."""
    if math.prod(_dims(case)) * case["ls"] > 1 << 16:
        return None
    if case["c12"]:
        U = _stored_links(dict(case, prec="fp64"), U)
    be, bo = b * (1 - odd), b * odd
    src = bo + 0.5 * _hop(U, _mooee(be, False, inverse=True), False) * odd
    rhs = _mpc(U, src, True, odd)
    x = torch.zeros_like(rhs)
    r = rhs.clone()
    p = r.clone()
    rr = r.abs().square().sum()
    stop = rr * 1e-26
    for it in range(2000):
        ap = _mpc(U, _mpc(U, p, False, odd), True, odd)
        alpha = rr / (p.conj() * ap).sum().real
        x = x + alpha * p
        r = r - alpha * ap
        new = r.abs().square().sum()
        if new <= stop:
            break
        p = r + (new / rr) * p
        rr = new
    xe = _mooee(be + 0.5 * _hop(U, x, False) * (1 - odd), False, inverse=True)
    return _device_layout(case, x + xe, dwf.FULL, "fp64")

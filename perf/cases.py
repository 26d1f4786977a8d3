"""Cases that stand for what a user of this library has it do, and the same results in plain torch at 64 bits.

A user keeps a hierarchy (a gauge field's operators, interpolations and coarse operators) on the device and
calls the C ABI through its Python binding with fields that are on the device: whole solves (one right-hand
side, a batch, a small FP64 one), and, in programs that build their own cycle or update a Monte Carlo chain,
the operator, the smoother of the fine and of a coarse level, the two transfers, and the rebuild of the
hierarchy after a change of the gauge field.  Lattices, aggregates, SAP blocks, test-vector counts and masses
are those of the repository's workloads and of its default parameters, and sizes between and around them.

Every state has a hierarchy of its own, on links and fields drawn from the seed: links U = exp(i eps H), H
traceless Hermitian with N(0,1) entries; fields complex N(0,1).  The building blocks run on hierarchies whose
test vectors are the caller's random fields (no smoothing, no setup cycles), so that P and the coarse
operators follow from the inputs in closed form; the solves run on a hierarchy set up by the library.
The fields are made on a stream of the user's own, which the handle is told to use (ddamg_set_stream), so
nothing has to be waited for between the torch operations and the library's kernels.

The values that `tolerance` states are about four times what the outputs were seen to be off the 64-bit results,
and at least 1e-6 in FP32 (other orders of summation, the tensor-core and the CUDA-core kernels).
"""
import math

import numpy as np
import torch

import paper_1307_6101_gb300 as dd

MASS = {0.3: -0.5132478239410015, 0.4: -0.6934846463376233}   # (eps, csw = 0 / 1) of the workloads
DEVICE = "cuda"
SETUP_SEED = 77                                              # random start vectors of the solves' setup


def listed():
    return [
        # one application of the outer operator to one field of the smallest workload: latency
        case("apply_f64_8", "apply", (8, 8, 8, 8), precision=0, agg=4, sap=2, n_tv=2),
        # the outer operator on a large lattice: the largest resident lattice of the serving workload but one
        case("apply_f64_24x48", "apply", (48, 24, 24, 24), precision=0, agg=4, sap=4, n_tv=2),
        # the smoother with the default parameters (FP32, 2^4 blocks) on a lattice of mixed extents, two fields
        case("smooth_f32_b2", "smooth", (24, 12, 20, 16), n=2, precision=1, agg=2, sap=2, n_tv=2, mr=3, its=5),
        # the smoother of the three-level workload (FP16 storage, 4^4 blocks), one field: one call of a K-cycle
        case("smooth_f16_b4", "smooth", (32, 16, 16, 16), precision=2, agg=4, sap=4, n_tv=2, mr=4, its=5),
        # the same for a batch of twelve, as in a propagator calculation
        case("smooth_f16_b4_r12", "smooth", (32, 16, 16, 16), n=12, precision=2, agg=4, sap=4, n_tv=2, mr=4, its=5),
        # the smoother on the first coarse level (40 dof, 2^4 blocks), one field
        case("smooth_l1", "smooth", (32, 16, 16, 16), precision=2, level=1, levels=3, agg=4, sap=4, n_tv=20, mr=4,
             its=5),
        # restriction and interpolation between the fine and the first coarse level, one field
        case("transfer", "transfer", (32, 16, 16, 16), precision=2, agg=4, sap=4, n_tv=20),
        # and a batch of twelve
        case("transfer_r12", "transfer", (32, 16, 16, 16), n=12, precision=2, agg=4, sap=4, n_tv=20),
        # a step of a Monte Carlo chain: a new gauge field into a three-level hierarchy, its coarse operators
        case("rebuild", "rebuild", (32, 16, 16, 16), precision=2, levels=3, agg=4, sap=4, n_tv=20, mr=4),
        # a small two-level FP64 solve (8^4, plain Wilson): latency
        case("solve_f64_8", "solve", (8, 8, 8, 8), precision=0, agg=4, sap=2, n_tv=8, eps=0.3, mr=4, nu=3, n_inv=3,
             restart=25),
        # the headline: a three-level mixed-precision solve for one right-hand side
        case("solve_mixed", "solve", (32, 16, 16, 16), precision=2, levels=3, agg=4, sap=4, n_tv=20, mr=4, nu=5,
             n_inv=2, restart=10),
        # twelve right-hand sides in one batch: a propagator
        case("solve_mixed_r12", "solve", (32, 16, 16, 16), n=12, precision=2, levels=3, agg=4, sap=4, n_tv=20, mr=4,
             nu=5, n_inv=2, restart=10),
    ]


def case(name, op, dims, n=1, precision=0, level=0, levels=2, agg=4, sap=4, n_tv=2, eps=0.4, mr=3, nu=5, its=1,
         n_inv=0, restart=10):
    c = dict(op=op, T=dims[0], Z=dims[1], Y=dims[2], X=dims[3], n=n, precision=precision, level=level, levels=levels,
             agg=agg, sap=sap, n_tv=n_tv, eps=eps, mr=mr, nu=nu, its=its, n_inv=n_inv, restart=restart)
    return dict(c, name=name) if name else c


def draw(rng):
    """A case of the ranges above: any of the calls, lattices from 8^4 up, every precision, one to twelve fields."""
    op = rng.choice(["apply", "smooth", "smooth", "smooth", "transfer", "transfer", "rebuild", "solve", "solve"])
    precision = rng.choice([0, 1, 2, 2, 2])
    b = rng.choice([2, 3, 4, 4])
    step = 2 * b   # an even number of blocks per direction, even coarse extents

    def lattice(lo, hi):
        """About exp(uniform(log lo, log hi)) sites, extents multiples of `step`, time the longest."""
        want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        side = want ** 0.25
        for _ in range(1000):
            d = [max(1, round(side * math.exp(rng.uniform(-0.35, 0.35)) / step)) * step for _ in range(4)]
            if lo <= math.prod(d) <= hi:
                break
        else:
            d = [step * (2 if step < 8 else 1)] * 4
        return sorted(d, reverse=True)[:1] + sorted(d)[:3]

    if op == "apply":
        n = rng.choice([1, 1, 2, 3, 5])
        return case("", op, lattice(1200, 660000 // n), n=n, precision=precision, agg=b, sap=b, n_tv=2)
    if op == "smooth" and rng.random() < 0.35:   # a coarse level
        return case("", op, (rng.choice([16, 32]), 16, 16, 16), n=rng.choice([1, 1, 2, 3, 4]),
                    precision=rng.choice([1, 2, 2]), level=1, levels=3, n_tv=rng.choice([8, 12, 20, 20]), mr=rng.choice([3, 4]),
                    its=rng.choice([1, 3, 5]))
    if op == "smooth":
        n = rng.choice([1, 1, 2, 4, 7, 12]) if precision else 1
        return case("", op, lattice(1200, 130000 // (1 if precision else 4)), n=n, precision=precision, agg=b, sap=b, n_tv=2,
                    mr=rng.choice([3, 4]), its=rng.choice([1, 2, 5]))
    if op == "transfer":
        n = rng.choice([1, 1, 2, 4, 7, 12]) if precision else rng.choice([1, 2])
        n_tv = min(rng.choice([4, 8, 12, 20, 24, 28]), 12 if b == 2 else 28)
        return case("", op, lattice(4000, 130000), n=n, precision=precision, agg=b, sap=b, n_tv=n_tv)
    if op == "rebuild":
        return case("", op, (16 * rng.choice([1, 2]), 16, 16, 16), precision=rng.choice([1, 2]), levels=3, agg=4, sap=4,
                    n_tv=rng.choice([8, 12, 20]), mr=4)
    if precision == 0:
        return case("", "solve", (8 * rng.choice([1, 2]), 8, 8, 8), n=rng.choice([1, 2]), precision=0, agg=4,
                    sap=rng.choice([2, 4]), n_tv=rng.choice([6, 8, 12]), eps=rng.choice([0.3, 0.4]), mr=rng.choice([3, 4]), nu=3,
                    n_inv=2, restart=rng.choice([10, 25]))
    sap = rng.choice([2, 4, 4])
    n = rng.choice([1, 2, 3, 6, 12] if precision == 2 and sap == 4 else [1, 2, 3])
    return case("", "solve", (16 * rng.choice([1, 2]), 16, 16, 16), n=n, precision=precision, levels=3, agg=4, sap=sap,
                n_tv=rng.choice([16, 20]), mr=rng.choice([3, 4]), nu=5, n_inv=rng.choice([1, 2]), restart=10)


# ---- inputs ---------------------------------------------------------------------------------------------------


def _dims(c):
    return c["T"], c["Z"], c["Y"], c["X"]


def _csw(c):
    return 0.0 if c["eps"] == 0.3 else 1.0


def _levels(c):
    """(dims, dof) per level; aggregates below the first are 2^4."""
    out, d, n = [], _dims(c), 12
    for l in range(c["levels"]):
        out.append((d, n))
        d = tuple(x // (c["agg"] if l == 0 else 2) for x in d)
        n = 2 * _n_tv(c, l)
    return out


def _n_tv(c, l):
    """20 test vectors above 28, as the workloads have them."""
    return c["n_tv"] if l == 0 else min(28, c["n_tv"] + 8)


def _field(gen, *shape):
    return torch.view_as_complex(torch.randn(*shape, 2, generator=gen, dtype=torch.float64, device=DEVICE))


def _links(gen, dims, eps):
    """U[t, z, y, x, mu, 3, 3] = exp(i eps H) by scaling and squaring, re-unitarised."""
    a = _field(gen, *dims, 4, 3, 3)
    h = 0.5 * (a + a.mH)
    h = h - (torch.diagonal(h, dim1=-2, dim2=-1).sum(-1) / 3.0)[..., None, None] * torch.eye(3, device=DEVICE)
    h = (1j * eps / 16.0) * h
    u = torch.eye(3, dtype=torch.complex128, device=DEVICE).expand_as(h).clone()
    for k in range(14, 0, -1):
        u = _mm(h, u) / k
        torch.diagonal(u, dim1=-2, dim2=-1).add_(1.0)
    for _ in range(4):
        u = _mm(u, u)
    r0 = u[..., 0, :] / torch.linalg.vector_norm(u[..., 0, :], dim=-1, keepdim=True)
    r1 = u[..., 1, :]
    r1 = r1 - (r0.conj() * r1).sum(-1, keepdim=True) * r0
    r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
    r2 = torch.stack([r0[..., 1] * r1[..., 2] - r0[..., 2] * r1[..., 1], r0[..., 2] * r1[..., 0] - r0[..., 0] * r1[..., 2],
                      r0[..., 0] * r1[..., 1] - r0[..., 1] * r1[..., 0]], -1).conj()
    return torch.stack([r0, r1, r2], -2).contiguous()


def _mm(a, b):
    """3x3 products as sums of broadcast columns."""
    return a[..., :, 0:1] * b[..., 0:1, :] + a[..., :, 1:2] * b[..., 1:2, :] + a[..., :, 2:3] * b[..., 2:3, :]


def _inputs(c, seed):
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(1000003 * int(seed) + 17)
    lv = _levels(c)
    s = {"U": _links(gen, _dims(c), c["eps"])}
    if c["op"] != "solve":
        s["tv"] = [_field(gen, _n_tv(c, 0), *_dims(c), 12)]
        for l in range(1, c["levels"] - 1):
            s["tv"].append(_field(gen, _n_tv(c, l) - _n_tv(c, l - 1), *lv[l][0], lv[l][1]) if _n_tv(c, l) > _n_tv(c, l - 1)
                           else None)
    d, n = lv[c["level"]]
    if c["op"] == "rebuild":
        s["U1"] = _links(gen, _dims(c), c["eps"])
    else:
        s["b"] = _field(gen, c["n"], *d, n)
    if c["op"] == "smooth":
        s["z0"] = 0.2 * _field(gen, c["n"], *d, n)
    if c["op"] == "transfer":
        s["phi"] = _field(gen, c["n"], *lv[1][0], lv[1][1])
    return s


def prepare(c, seed):
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        s = _inputs(c, seed)
        stream.synchronize()
        L = c["levels"]
        a, b = c["agg"], c["sap"]
        p = dd.ddamg_default_params(
            levels=L, agg=[(a,) * 4] + [(2,) * 4] * (L - 2), n_tv=[_n_tv(c, l) for l in range(L - 1)],
            sap_block=[(b,) * 4] + [(2,) * 4] * (L - 2), mr_steps=c["mr"], nu=c["nu"], n_inv=c["n_inv"],
            eta_passes=3 if c["op"] == "solve" else 0, outer_restart=c["restart"], precision=c["precision"],
            max_rhs=c["n"], seed=SETUP_SEED)
        h = dd.ddamg_setup(s["U"], _dims(c), -1, MASS[c["eps"]], _csw(c), p, s.get("tv"))
        dd.ddamg_set_stream(h, stream.cuda_stream)
        lv = _levels(c)
        prec = 1 if c["precision"] else 0
        st = {"c": c, "h": h, "stream": stream, "prec": prec}
        st.update({k: s[k] for k in ("b", "z0", "phi", "U1") if k in s})
        if c["op"] in ("apply", "solve"):
            st["x"] = torch.empty_like(s["b"])
        if c["op"] == "transfer":
            st["coarse"], st["fine"] = torch.empty_like(s["phi"]), torch.empty_like(s["b"])
        if c["op"] == "rebuild":
            st["D"] = [torch.empty(*d, 9, n, n, dtype=torch.complex128, device=DEVICE) for d, n in lv[1:]]
        stream.synchronize()
    return st


def run(s):
    c, h, n = s["c"], s["h"], s["c"]["n"]
    with torch.cuda.stream(s["stream"]):
        if c["op"] == "apply":
            dd.ddamg_apply(h, 0, s["prec"], s["b"], s["x"], n)
            return s["x"]
        if c["op"] == "smooth":
            z = s["z0"].clone()
            dd.ddamg_smooth(h, c["level"], s["prec"], s["b"], z, n, c["its"])
            return z
        if c["op"] == "transfer":
            dd.ddamg_restrict(h, 0, s["prec"], s["b"], s["coarse"], n)
            dd.ddamg_prolong(h, 0, s["prec"], s["phi"], s["fine"], n)
            return {"coarse": s["coarse"], "fine": s["fine"]}
        if c["op"] == "rebuild":
            dd.ddamg_update_gauge(h, s["U1"], 0)
            for l, D in enumerate(s["D"]):
                dd.ddamg_get_coarse_operator(h, l + 1, D)
            return s["D"]
        st = dd.ddamg_solve(h, s["b"], s["x"], n, 1e-10, raise_noconv=True)
        assert all(r["converged"] for r in st)
        return s["x"]


def work(c):
    """Bytes: fields in the ABI's FP64 once in and once out, operator data once in its stored format.  Flops: the
    products and sums of the method (an FMA is two) for the steps that the parameters ask for."""
    V = math.prod(_dims(c))
    n, n_tv = c["n"], c["n_tv"]
    link = {0: 16, 1: 8, 2: 4}[c["precision"]]
    D = 8 * (12 + 2 * 66 + 24) + 2 * (12 + 15 * 16) + 48   # the fine operator per site (hops, clover term, combination)
    lv = _levels(c)
    if c["op"] == "apply":
        return {"bytes": V * (n * 2 * 192 + 36 * link + 36 * link), "flops": V * n * D}
    if c["op"] == "smooth" and c["level"] == 0:
        return {"bytes": V * (n * 3 * 192 + 72 * link), "flops": V * n * c["its"] * (D + c["mr"] * (D + 120 + 192))}
    if c["op"] == "smooth":
        d, k = lv[1]
        vc, inside = math.prod(d), 5   # a site of a 2^4 block has four neighbours in it
        return {"bytes": vc * (n * 3 * 16 * k + 9 * k * k * link),
                "flops": vc * n * c["its"] * 8 * k * k * (9 + c["mr"] * inside)}
    if c["op"] == "transfer":
        vc, k = math.prod(lv[1][0]), lv[1][1]
        return {"bytes": V * (n * 2 * 192 + 12 * n_tv * link) + vc * n * 2 * k * 16, "flops": V * n * 2 * 12 * n_tv * 8}
    if c["op"] == "rebuild":
        by, fl = V * 36 * 16, 0
        for l in range(c["levels"] - 1):
            (d, m), (dc, k) = lv[l], lv[l + 1]
            v, vc, N = math.prod(d), math.prod(dc), _n_tv(c, l)
            by += v * m * N * 16 * 2 + vc * 9 * k * k * 16
            fl += v * m * N * N * 16                                    # two passes of Gram-Schmidt
            fl += v * 2 * N * (D if l == 0 else 9 * 8 * m * m)          # D on the columns of P by chirality
            fl += 8 * v * m * N * 2 * N * 2                              # the products with P^dagger (faces and interior)
        return {"bytes": by, "flops": fl}
    # a solve: fields and the operators of all levels once; an outer iteration's operator, Gram-Schmidt and smoother
    # for the iterations that 1e-10 takes (about fifteen)
    by, fl, its = V * (n * 2 * 192 + 72 * 16 + 72 * link), 0, 15
    for l in range(c["levels"] - 1):
        (d, m), (dc, k) = lv[l], lv[l + 1]
        v, vc = math.prod(d), math.prod(dc)
        by += v * m * _n_tv(c, l) * link + vc * 9 * k * k * link
        fl += v * m * _n_tv(c, l) * 16
        fl += v * c["nu"] * ((D + c["mr"] * (D + 312)) if l == 0 else 8 * m * m * (9 + 5 * c["mr"]))
    return {"bytes": by, "flops": n * its * (fl + V * (D + 12 * 8 * 4 * 5))}


def tolerance(c):
    if c["op"] == "solve":
        return {"rel": 2e-9}          # both sides stop at a relative residual of 1e-10; sigma_min is about 0.07
    if c["precision"] == 0:
        return {"rel": 2e-15} if c["op"] in ("apply", "transfer") else {"rel": 1e-14}
    if c["level"] == 1 and c["precision"] == 2:
        return {"rel": 2e-5}          # the blocks are FP32 products rounded to FP16: another order rounds some the other way
    return {"rel": 1e-6}              # FP32 sums of up to some thousand products, chained over a few sweeps


# ---- the same in plain torch, 64 bits -----------------------------------------------------------------------------

_SIGMA = [[[1, 0], [0, -1]], [[0, -1j], [1j, 0]], [[0, 1], [1, 0]]]   # of the directions z, y, x


def _gamma(mu):
    g = torch.zeros(4, 4, dtype=torch.complex128)
    if mu == 0:
        g[:2, 2:] = g[2:, :2] = torch.eye(2, dtype=torch.complex128)
    else:
        s = torch.tensor(_SIGMA[mu - 1], dtype=torch.complex128)
        g[:2, 2:], g[2:, :2] = -1j * s, 1j * s
    return g.to(DEVICE)


def _half(x):
    """Rounded to the nearest FP16 numbers (numpy rounds FP64 once; torch goes by way of FP32)."""
    r = torch.view_as_real(x.resolve_conj().contiguous()).cpu().numpy().astype(np.float16).astype(np.float64)
    return torch.view_as_complex(torch.from_numpy(r)).to(x.device)


class _Fine:
    """The Wilson-clover operator; precision 2: links and clover term rounded to FP16, as the storage format says."""

    def __init__(self, U, m0, csw, half):
        self.dims, self.n = U.shape[:4], 12
        A = self.clover(U, csw)
        shift = m0 + 4.0
        if half:
            U, A, shift = _half(U), _half(A), float(np.float32(shift))
        self.A = A + shift * torch.eye(6, dtype=torch.complex128, device=DEVICE)   # [..., chirality, 6, 6]
        self.U = [U[..., mu, :, :] for mu in range(4)]
        self.Ub = [torch.roll(u, 1, mu).mH for mu, u in enumerate(self.U)]
        self.spin = []
        for mu in range(4):
            g = _gamma(mu)
            perm = [int(g[s].abs().argmax()) for s in range(4)]
            self.spin.append((perm, torch.stack([g[s, perm[s]] for s in range(4)])[:, None]))

    @staticmethod
    def clover(U, csw):
        C = torch.zeros(*U.shape[:4], 12, 12, dtype=torch.complex128, device=DEVICE)

        def at(v, mu, d):
            return torch.roll(v, -d, mu)

        if csw:
            u = [U[..., m, :, :] for m in range(4)]
            for m in range(4):
                for n in range(m + 1, 4):
                    # the four leaves of the plane: closed paths from x around x +- m, x +- n, in the same sense
                    um, un = u[m], u[n]
                    q = _mm(_mm(um, at(un, m, 1)), _mm(un, at(um, n, 1)).mH)
                    q = q + _mm(_mm(un, at(at(um, n, 1), m, -1).mH), _mm(at(un, m, -1).mH, at(um, m, -1)))
                    q = q + _mm(_mm(at(at(un, m, -1), n, -1), at(um, m, -1)).mH, _mm(at(at(um, m, -1), n, -1), at(un, n, -1)))
                    q = q + _mm(_mm(at(un, n, -1).mH, at(um, n, -1)), _mm(at(at(un, n, -1), m, 1), um.mH))
                    f = q - q.mH
                    C += torch.einsum("st,...ab->...satb", _gamma(m) @ _gamma(n), f).reshape(C.shape)
        C = -(csw / 16.0) * C
        return torch.stack([C[..., :6, :6], C[..., 6:, 6:]], -3)

    def diag(self, psi):
        v = psi.reshape(*psi.shape[:-1], 2, 6)
        out = self.A[..., :, 0] * v[..., 0:1]
        for j in range(1, 6):
            out = out + self.A[..., :, j] * v[..., j:j + 1]
        return out.reshape(psi.shape)

    def hop(self, psi, mu, d):
        """-1/2 (1 -+ gamma_mu) U psi(x +- mu), antiperiodic in time."""
        v = torch.roll(psi, -d, 1 + mu).reshape(*psi.shape[:-1], 4, 3)
        if mu == 0:
            v[:, -1 if d > 0 else 0] *= -1
        u = self.U[mu] if d > 0 else self.Ub[mu]
        w = u[..., None, :, 0] * v[..., 0:1] + u[..., None, :, 1] * v[..., 1:2] + u[..., None, :, 2] * v[..., 2:3]
        perm, ph = self.spin[mu]
        return (-0.5 * (w - d * ph * w[..., perm, :])).reshape(psi.shape)


class _Coarse:
    """The 9-point stencil of blocks blk[..., k, row, column] (k: self, forward t z y x, backward)."""

    def __init__(self, blk, half):
        self.dims, self.n = blk.shape[:4], blk.shape[-1]
        if half:
            s = torch.view_as_real(blk).abs().amax((-1, -2, -3, -4)).float().double()[..., None, None, None]
            blk = _half(blk / s) * s
        self.blk = blk

    def diag(self, phi):
        return torch.einsum("tzyxij,ntzyxj->ntzyxi", self.blk[..., 0, :, :], phi)

    def hop(self, phi, mu, d):
        return torch.einsum("tzyxij,ntzyxj->ntzyxi", self.blk[..., 1 + mu if d > 0 else 5 + mu, :, :], torch.roll(phi, -d, 1 + mu))


def _inside(dims, tile, mu, d):
    """Whether the hop x -> x + d mu stays in x's tile, as a mask over the lattice."""
    c = torch.arange(dims[mu], device=DEVICE)
    m = ((c + d) % dims[mu]) // tile[mu] == c // tile[mu]
    return m.double().reshape([-1 if k == mu else 1 for k in range(4)] + [1])


def _apply(op, v, tile=None):
    """op v; with tile, the hops that leave a tile are dropped."""
    out = op.diag(v)
    for mu in range(4):
        for d in (1, -1):
            w = op.hop(v, mu, d)
            out = out + (w if tile is None else _inside(op.dims, tile, mu, d) * w)
    return out


def _widen(dims, b):
    """SAP blocks: the smallest extents of at least b that give an even number of blocks, or one block."""
    out = []
    for L in dims:
        e = b
        while e < L and (L % e or (L // e) % 2):
            e += 1
        out.append(min(e, L))
    return out


def _smooth(op, b, z, tile, mr, its):
    dims = op.dims
    shape = [b.shape[0]] + [x for L, t in zip(dims, tile) for x in (L // t, t)] + [op.n]

    def block_sum(v):
        return v.reshape(shape).sum((2, 4, 6, 8, 9), keepdim=True).expand(shape).reshape(v.shape)

    col = sum((torch.arange(L, device=DEVICE) // t).reshape([-1 if k == mu else 1 for k in range(4)])
              for mu, (L, t) in enumerate(zip(dims, tile))) % 2
    for _ in range(its):
        for colour in (0, 1):
            r = (b - _apply(op, z)) * (col == colour)[..., None]
            for _ in range(mr):
                p = _apply(op, r, tile)
                den = block_sum(p.real ** 2 + p.imag ** 2)
                alpha = torch.where(den > 0, block_sum(p.conj() * r) / den.clamp(min=1e-300), 0.0)
                z = z + alpha * r
                r = r - alpha * p
    return z


class _Transfer:
    """P from fields V[j], orthonormalised per aggregate and chirality (first column first)."""

    def __init__(self, V, agg, half):
        self.N, self.dims, self.n = V.shape[0], V.shape[1:5], V.shape[5]
        self.agg = agg
        self.cdims = tuple(L // agg for L in self.dims)
        M = self.split(V)                                              # [aggregates, 2, rows, N]
        G = M.mH @ M
        R = torch.linalg.cholesky(G).mH
        self.R = R
        P = torch.linalg.solve_triangular(R, M, upper=True, left=False)
        if half:
            s = torch.view_as_real(P).abs().amax((-1, -2, -3)).float().double()[..., None, None]
            self.Q = _half(P / s) * s
        else:
            self.Q = P
        self.P = P

    def split(self, v):
        """[n, T, Z, Y, X, dof] -> [aggregates, 2, rows of one chirality, n]."""
        a = self.agg
        v = v.reshape(v.shape[0], *[x for L in self.cdims for x in (L, a)], 2, self.n // 2)
        return v.permute(1, 3, 5, 7, 9, 2, 4, 6, 8, 10, 0).reshape(math.prod(self.cdims), 2, a ** 4 * self.n // 2, v.shape[0])

    def join(self, m):
        a, k = self.agg, m.shape[-1]
        m = m.reshape(*self.cdims, 2, a, a, a, a, self.n // 2, k)
        return m.permute(10, 0, 5, 1, 6, 2, 7, 3, 8, 4, 9).reshape(k, *self.dims, self.n)

    def restrict(self, v, P=None):
        y = (self.Q if P is None else P).mH @ self.split(v)              # [aggregates, 2, N, n]
        return y.permute(3, 0, 1, 2).reshape(v.shape[0], *self.cdims, 2 * self.N)

    def prolong(self, phi, P=None):
        y = phi.reshape(phi.shape[0], -1, 2, self.N).permute(1, 2, 3, 0)
        return self.join((self.Q if P is None else P) @ y)

    def galerkin(self, op):
        """The blocks of P^dagger op P."""
        nc = 2 * self.N
        blk = torch.zeros(*self.cdims, 9, nc, nc, dtype=torch.complex128, device=DEVICE)
        tile = [self.agg] * 4
        F = self.join(self.P)                                            # the N columns as fields
        for s in range(2):
            keep = torch.zeros(self.n, device=DEVICE, dtype=torch.float64)
            keep[s * self.n // 2:(s + 1) * self.n // 2] = 1.0
            for j in range(self.N):
                v = F[j:j + 1] * keep
                col = s * self.N + j
                selfpart = op.diag(v)
                for mu in range(4):
                    for d in (1, -1):
                        w, m = op.hop(v, mu, d), _inside(self.dims, tile, mu, d)
                        selfpart = selfpart + m * w
                        blk[..., (1 if d > 0 else 5) + mu, :, col] = self.restrict((1.0 - m) * w, self.P)[0]
                blk[..., 0, :, col] = self.restrict(selfpart, self.P)[0]
        return blk


def _chain(c, s, U, half, depth):
    """The fine operator, then per level (transfer, Galerkin blocks) down to `depth` levels below it, from the test vectors."""
    op = _Fine(U, MASS[c["eps"]], _csw(c), False)   # the Galerkin products are formed from the unrounded operators
    tv, out = s["tv"][0], []
    for l in range(depth):
        t = _Transfer(tv, c["agg"] if l == 0 else 2, half)
        blk = t.galerkin(op)
        out.append((t, blk))
        if l + 1 < depth:
            tv = t.restrict(tv, t.P)
            if s["tv"][l + 1] is not None:
                tv = torch.cat([tv, s["tv"][l + 1]])
            op = _Coarse(blk, False)
    return out


def _cgnr(op, b, tol, most):
    """D x = b by conjugate gradients on D^dagger D, D^dagger = Gamma_5 D Gamma_5."""
    g5 = torch.ones(12, dtype=torch.float64, device=DEVICE)
    g5[6:] = -1.0

    def dot(u):
        return (u.real ** 2 + u.imag ** 2).sum((1, 2, 3, 4, 5), keepdim=True)

    x, s = torch.zeros_like(b), b.clone()
    r = g5 * _apply(op, g5 * s)
    p, gam, goal = r, dot(r), tol * tol * dot(b)
    for k in range(most):
        q = _apply(op, p)
        al = gam / dot(q)
        x, s = x + al * p, s - al * q
        r = g5 * _apply(op, g5 * s)
        new = dot(r)
        p, gam = r + (new / gam) * p, new
        if k % 16 == 15 and bool((dot(s) <= goal).all()):
            break
    return x


def exact(c, seed):
    s = _inputs(c, seed)
    half, m0 = c["precision"] == 2, MASS[c["eps"]]
    if c["op"] == "apply":
        return _apply(_Fine(s["U"], m0, _csw(c), half), s["b"])
    if c["op"] == "smooth" and c["level"] == 0:
        return _smooth(_Fine(s["U"], m0, _csw(c), half), s["b"], s["z0"], _widen(_dims(c), c["sap"]), c["mr"], c["its"])
    if c["op"] == "smooth":
        (_, blk), = _chain(c, s, s["U"], half, 1)
        return _smooth(_Coarse(blk, half), s["b"], s["z0"], _widen(_levels(c)[1][0], 2), c["mr"], c["its"])
    if c["op"] == "transfer":
        t = _Transfer(s["tv"][0], c["agg"], half)
        return {"coarse": t.restrict(s["b"]), "fine": t.prolong(s["phi"])}
    if c["op"] == "rebuild":
        # the test vectors are those that the setup left on the first gauge field: P does not depend on the links here
        return [blk for _, blk in _chain(c, s, s["U1"], half, c["levels"] - 1)]
    if c["n"] * math.prod(_dims(c)) > 200000:
        return None   # a minute or more of conjugate gradients
    return _cgnr(_Fine(s["U"], m0, _csw(c), False), s["b"], 1e-13, 4000)

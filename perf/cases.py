"""The workloads by which the speed of this framework is judged.

A case is one call (or one forward and backward pass) that a program using the
package makes on one lattice: the stencil apply in each precision, the link
precompute, the differentiable operator, the pseudofermion action, mixed and
batched solves, and the overlap operator.  Lattices are those of the package's
own workloads (8^4, 12^4, 16^3x32, 24^3x48, 32^3x64), a ragged one, and, in
draw(), any extents from 4 to 64.

``exact`` gives the same results in plain torch (complex128): path averages over
the first step of every path, projection by an eigendecomposition, the stencil
hop by hop, BiCGstab, and a Chebyshev sign function.
"""
import itertools
import math

import torch

from paper_1012_3615_gb300 import Brillouin, DiracFunction, InverseActionFunction, synth

BC = (1, 1, 1, -1)  # antiperiodic in t
VMAX = 32 * 32 * 32 * 64

# stored bytes of one hopping field entry set per site
LINK_BYTES = {("f64", "full"): 144, ("f32", "full"): 72, ("f32", "2row"): 48, ("f32", "8param"): 32,
              ("f16", "full"): 36, ("f16", "2row"): 24, ("f16", "8param"): 16}
SITE_FLOPS = 29208  # of one apply, per site and right-hand side: 80 colour products on 4 spins and the class sums


def _case(name, kind, L, **more):
    c = {"name": name, "kind": kind, "x": L[0], "y": L[1], "z": L[2], "t": L[3], "eps": 0.3, "m0": 0.0}
    c.update(more)
    return c


def listed():
    return [
        # the operator on the largest lattice of the bandwidth sweep: the inner apply of a propagator solve
        _case("apply_f32_32x32x32x64", "apply", (32, 32, 32, 64), prec="f32", comp="full", nrhs=1, op="D", csw=0.0),
        # the smallest call: one FP64 apply on 8^4, where latency and idle SMs count
        _case("apply_f64_8x8x8x8", "apply", (8, 8, 8, 8), prec="f64", comp="full", nrhs=1, op="D", csw=0.0),
        # FP64 D^dagger on the mixed-solve lattice: the true residuals, normal equations and gradients
        _case("adjoint_f64_16x16x16x32", "apply", (16, 16, 16, 32), prec="f64", comp="full", nrhs=1, op="Ddag",
              csw=0.0, eps=0.4, m0=-0.05),
        # 12 spin-colour components together on half-precision 2-row fields: the apply of a batched propagator
        _case("apply_f16_24x24x24x48_n12", "apply", (24, 24, 24, 48), prec="f16", comp="2row", nrhs=12, op="D",
              csw=0.0, eps=0.35),
        # the hermitian overlap kernel on odd extents, a few vectors: nothing divides a warp or a tile
        _case("overlap_kernel_f32_13x9x11x21_n3", "apply", (13, 9, 11, 21), prec="f32", comp="2row", nrhs=3, op="H",
              csw=0.0),
        # the clover-improved operator at tree level (c_SW = 1)
        _case("clover_f32_16x16x16x32", "apply", (16, 16, 16, 32), prec="f32", comp="full", nrhs=1, op="D", csw=1.0,
              eps=0.4),
        # hopping fields of a new gauge configuration, with the copy that a mixed solve reads
        _case("build_16x16x16x32", "build", (16, 16, 16, 32), prec="f32", comp="2row", eps=0.4),
        # a differentiable apply: forward, and gradients in the links and the spinor
        _case("dirac_12x12x12x12", "dirac", (12, 12, 12, 12)),
        # pseudofermion action and force, as one molecular-dynamics step needs them (two FP64 solves)
        _case("action_12x12x12x12", "action", (12, 12, 12, 12), m0=0.1, tol=1e-12),
        # one propagator component by FP64 defect correction around FP32
        _case("solve_mixed_16x16x16x32", "solve", (16, 16, 16, 32), prec="f32", comp="2row", mode=1, nrhs=1, eps=0.4,
              m0=-0.05, tol=1e-12),
        # a whole point-source propagator: 12 right-hand sides advance together
        _case("solve_batched_16x16x16x32_n12", "solve", (16, 16, 16, 32), prec="f32", comp="2row", mode=4, nrhs=12,
              eps=0.35, m0=0.0, tol=1e-12),
        # the overlap operator with an FP32 sign polynomial, after its setup
        _case("overlap_12x12x12x12", "overlap", (12, 12, 12, 12), prec="f32", comp="full", nlow=4, nrhs=1),
    ]


def _extents(rng, vmin, vmax):
    """four extents of a volume spread over [vmin, vmax] on a logarithmic scale; about half of the lattices have an
    x extent of the usual production sizes, the rest take any"""
    while True:
        side = math.exp(rng.uniform(math.log(vmin), math.log(vmax))) ** 0.25
        L = [max(4, min(64, round(side * math.exp(rng.uniform(-0.45, 0.45))))) for _ in range(4)]
        if rng.random() < 0.5:
            L[0] = rng.choice([8, 12, 16, 24, 32])
        if vmin <= L[0] * L[1] * L[2] * L[3] <= vmax:
            return L


def draw(rng):
    kind = rng.choice(["apply"] * 6 + ["build", "dirac", "action", "solve", "solve", "overlap"])
    eps = round(rng.uniform(0.25, 0.4), 3)
    if kind == "apply":
        prec, comp = rng.choice(sorted(LINK_BYTES) + [("f32", "full"), ("f32", "2row"), ("f64", "full")])
        nrhs = rng.choice([1, 1, 1, 2, 4, 5, 12])
        top = (VMAX // 8 if prec == "f64" else VMAX * 3) // nrhs
        L = _extents(rng, 256, min(VMAX, top))
        c = {"prec": prec, "comp": comp, "nrhs": nrhs, "op": rng.choice(["D", "D", "Ddag", "H"]),
             "csw": 1.0 if rng.random() < 0.15 else 0.0}
    elif kind == "build":
        L = _extents(rng, 1024, VMAX // 8)
        prec, comp = rng.choice(sorted(LINK_BYTES))
        c = {"prec": prec, "comp": comp}
    elif kind in ("dirac", "action"):
        L = _extents(rng, 256, 12 ** 4)
        c = {"m0": 0.1, "tol": 1e-12} if kind == "action" else {}
    elif kind == "solve":
        mode = rng.choice([0, 1, 2, 3, 4])
        nrhs = rng.choice([2, 5, 12]) if mode >= 3 else 1
        L = _extents(rng, 1024, (VMAX // 64 if mode == 0 else VMAX // 16))
        c = {"prec": "f32" if mode in (0, 1, 4) else "f16", "comp": rng.choice(["full", "2row"]), "mode": mode,
             "nrhs": nrhs, "m0": 0.0, "tol": 1e-12}
    else:
        L = _extents(rng, 256, 12 ** 4)
        c = {"prec": "f32", "comp": rng.choice(["full", "2row"]), "nlow": rng.choice([0, 2, 4]), "nrhs": rng.choice([1, 1, 2])}
    case = {"kind": kind, "x": L[0], "y": L[1], "z": L[2], "t": L[3], "eps": eps, "m0": 0.0}
    case.update(c)
    return case


def _lattice(c):
    return (c["x"], c["y"], c["z"], c["t"])


def _spinor_dtype(c):
    return torch.complex128 if c["prec"] == "f64" else torch.complex64


def _inputs(c, seed):
    """the links and the spinors of a case, the same for every implementation"""
    L, kind, n = _lattice(c), c["kind"], c.get("nrhs", 1)
    U = synth.random_su3_links_torch(L, c["eps"], 2 * seed + 1, device="cuda")
    if kind == "build":
        return U, None
    if kind == "apply":
        return U, synth.gaussian_spinor_torch(L, n, 2 * seed + 2, dtype=_spinor_dtype(c))
    if kind == "solve":
        g = torch.Generator(device="cuda")
        g.manual_seed(2 * seed + 2)
        V = synth.volume(L)
        if n == 1:  # Z2 noise
            z = torch.randint(0, 2, (1, V, 4, 3), generator=g, device="cuda") * 2 - 1
            return U, z.to(torch.complex128)
        b = torch.zeros((n, V, 12), dtype=torch.complex128, device="cuda")  # point sources, one per spin and colour
        at = int(torch.randint(0, V, (1,), generator=g, device="cuda"))
        for r in range(n):
            b[r, at, r % 12] = 1.0
        return U, b.reshape(n, V, 4, 3)
    if kind == "dirac":
        return U, synth.gaussian_spinor_torch(L, 2, 2 * seed + 2)  # psi, and the gradient that comes from above
    return U, synth.gaussian_spinor_torch(L, n, 2 * seed + 2)


def prepare(c, seed):
    kind = c["kind"]
    U, v = _inputs(c, seed)
    op = Brillouin(_lattice(c), BC)
    s = {"case": c, "op": op}
    if kind == "build":
        s["U"] = U
    elif kind in ("dirac", "action"):
        s["U"] = U.requires_grad_(True)
        s["v"] = v[0].contiguous().requires_grad_(True)
        if kind == "dirac":
            s["above"] = v[1].contiguous()
    else:
        op.build_hops(U, prec=c["prec"], comp=c["comp"])
        s["v"] = v
        if c.get("csw"):
            op.set_clover(c["csw"])
        if kind == "overlap":
            s["setup"] = op.overlap_setup(rho=1.0, nlow=c["nlow"], eps=1e-7, max_krylov=1000, tol=1e-6, prec=c["prec"])
    return s


def run(s):
    c, op = s["case"], s["op"]
    kind = c["kind"]
    if kind == "apply":
        if c["op"] == "H":
            return op.overlap_kernel(s["v"], rho=1.0, prec=c["prec"])
        return op.apply(s["v"], m0=c["m0"], dagger=c["op"] == "Ddag", prec=c["prec"])
    if kind == "build":
        op.build_hops(s["U"], prec=c["prec"], comp=c["comp"])
        return op.hops()
    if kind == "dirac":
        out = DiracFunction.apply(s["U"], s["v"], op, c["m0"])
        dU, dpsi = torch.autograd.grad(out, (s["U"], s["v"]), grad_outputs=s["above"])
        return {"out": out.detach(), "dU": dU, "dpsi": dpsi}
    if kind == "action":
        S = InverseActionFunction.apply(s["U"], s["v"], op, c["m0"], c["tol"])
        dU, dphi = torch.autograd.grad(S, (s["U"], s["v"]))
        return {"S": S.detach(), "dU": dU, "dphi": dphi}
    if kind == "solve":
        return op.solve(s["v"], m0=c["m0"], tol=c["tol"], mode=c["mode"])[0]
    return op.overlap(s["v"], m=0.0)


def work(c):
    """what a pass cannot do without: fields and spinors once, and the arithmetic of the method; a solve and a sign
    function as the number of applies that these lattices take to converge"""
    V = synth.volume(_lattice(c))
    kind, n = c["kind"], c.get("nrhs", 1)
    one64 = (40 * 144 + 384) * V
    if kind == "apply":
        elt = 16 if c["prec"] == "f64" else 8
        clov = (36 * elt if c["csw"] else 0) * V
        flops = (SITE_FLOPS + (2 * 18 * 2 * 12 if c["csw"] else 0)) * V * n
        return {"bytes": 40 * LINK_BYTES[c["prec"], c["comp"]] * V + clov + 24 * elt * V * n, "flops": flops}
    # 104 products of 3x3 matrices for the 36 averages over paths, and 36 projections
    build = {"bytes": (576 + 2 * 5760) * V, "flops": (104 * 216 + 36 * 1000) * V}
    if kind == "build":
        if c["prec"] != "f64":
            build["bytes"] += 40 * LINK_BYTES[c["prec"], c["comp"]] * V
        return build
    # the gradient in the links runs the build's products backwards twice (both factors)
    force = {"bytes": (2 * 576 + 2 * 192 + 5760) * V, "flops": 3 * build["flops"]}
    if kind == "dirac":
        return {"bytes": (576 + 5760) * V + 2 * one64 + force["bytes"],
                "flops": build["flops"] + 2 * SITE_FLOPS * V + force["flops"]}
    if kind == "action":
        applies = 120
        return {"bytes": (576 + 5760) * V + applies * one64 + force["bytes"],
                "flops": build["flops"] + applies * SITE_FLOPS * V + force["flops"]}
    if kind == "solve":
        if c["mode"] == 0:
            return {"bytes": 150 * (5760 + 384 * n) * V, "flops": 150 * SITE_FLOPS * V * n}
        links = 40 * LINK_BYTES[c["prec"], c["comp"]]
        return {"bytes": (150 * (links + 192 * n) + 3 * (5760 + 384 * n)) * V, "flops": 153 * SITE_FLOPS * V * n}
    links = 40 * LINK_BYTES[c["prec"], c["comp"]]
    return {"bytes": 27 * (links + 192) * V * n, "flops": 27 * SITE_FLOPS * V * n}


# ---- the same in plain torch, complex128 ------------------------------------------------------------------------

OFFSETS = [d[::-1] for d in itertools.product((-1, 0, 1), repeat=4) if any(d)]
LAMBDA = [240 / 128, -8 / 128, -4 / 128, -2 / 128, -1 / 128]
RHO = [0, 64 / 432, 16 / 432, 4 / 432, 1 / 432]
# the one non-zero entry of each row of the four gamma matrices (hermitian chiral basis): column and value
GAMMA = [[(3, 1j), (2, 1j), (1, -1j), (0, -1j)], [(3, -1), (2, 1), (1, 1), (0, -1)],
         [(2, 1j), (3, -1j), (0, -1j), (1, 1j)], [(2, 1), (3, 1), (0, 1), (1, 1)]]


def _mm(a, b):
    return sum(a[..., :, k, None] * b[..., None, k, :] for k in range(3))


def _dag(a):
    return a.conj().transpose(-1, -2)


class _Lattice:
    def __init__(self, L):
        self.L = L
        self.V = synth.volume(L)
        self.x = torch.as_tensor(synth.coordinates(L), device="cuda")

    def at(self, d):
        """indices of x + d, and the fermion's phase on the way"""
        idx = torch.zeros(self.V, dtype=torch.int64, device="cuda")
        ph = torch.ones(self.V, dtype=torch.float64, device="cuda")
        stride = 1
        for mu in range(4):
            y = self.x[:, mu] + d[mu]
            if BC[mu] < 0 and d[mu]:
                ph = torch.where((y < 0) | (y >= self.L[mu]), -ph, ph)
            idx += stride * (y % self.L[mu])
            stride *= self.L[mu]
        return idx, ph


class _Project(torch.autograd.Function):
    """argmax over SU(3) of Re tr(A^dagger Y): Y = A Q diag(e^{i th} / s) Q^dagger with s sin(th) the same for the
    three singular values"""

    @staticmethod
    def forward(ctx, A):
        e, Q = torch.linalg.eigh(_mm(_dag(A), A))
        s = e.clamp_min(1e-300).sqrt()
        det = (A[..., 0, :] * torch.linalg.cross(A[..., 1, :], A[..., 2, :])).sum(-1)
        t = -torch.angle(det)
        k = torch.zeros_like(t)
        for _ in range(60):
            r = (k[..., None] / s).clamp(-1, 1)
            f = torch.asin(r).sum(-1) - t
            df = (1 / (s * s - (k * k)[..., None]).clamp_min(1e-30).sqrt()).sum(-1)
            k = torch.maximum(torch.minimum(k - f / df, s[..., 0]), -s[..., 0])
        th = torch.asin((k[..., None] / s).clamp(-1, 1))
        Y = _mm(_mm(A, Q) * (torch.polar(1 / s, th))[..., None, :], _dag(Q))
        Y = 1.5 * Y - 0.5 * _mm(Y, _mm(_dag(Y), Y))
        ctx.save_for_backward(Y, Q, s * torch.cos(th))
        return Y

    @staticmethod
    def backward(ctx, G):
        Y, Q, h = ctx.saved_tensors
        B = _mm(_dag(Q), _mm(_mm(_dag(G), Y), Q))
        P = 0.5 * (B - _dag(B))
        X = P * (2 / (h[..., :, None] + h[..., None, :]))
        p = torch.diagonal(P, dim1=-2, dim2=-1).imag
        p = p - p.mean(-1, keepdim=True)
        m = -(p / h).sum(-1, keepdim=True) / (1 / h).sum(-1, keepdim=True)
        X = X - torch.diag_embed(torch.diagonal(X, dim1=-2, dim2=-1)) + torch.diag_embed(1j * (p + m) / h)
        return -_mm(Y, _mm(Q, _mm(X, _dag(Q))))


def _canonical(d):
    return [v for v in d if v][-1] > 0


def _hops(lat, U):
    """the 40 fields whose last non-zero offset component is +1"""
    A = {}
    for n in range(1, 5):
        for d in OFFSETS:
            if sum(map(abs, d)) != n:
                continue
            acc = 0
            for mu in range(4):
                if not d[mu]:
                    continue
                e = [0, 0, 0, 0]
                e[mu] = d[mu]
                to = lat.at(e)[0]
                F = U[:, mu] if d[mu] > 0 else _dag(U[:, mu][to])
                rest = tuple(v - w for v, w in zip(d, e))
                acc = acc + (F if n == 1 else _mm(F, A[rest][to]))
            A[d] = acc / n
    W = {}
    for d in OFFSETS:
        if _canonical(d):
            W[d] = A[d] if sum(map(abs, d)) == 1 else torch.cat([_Project.apply(a) for a in A[d].split(1 << 15)])
    return W


def _apply(lat, W, psi, m0, clover=None):
    """D psi for one field (V, 4, 3)"""
    out = (m0 + LAMBDA[0]) * psi
    for d, w in W.items():
        n = sum(map(abs, d))
        to, ph = lat.at(d)
        back, phb = lat.at([-v for v in d])
        for sign, chi in ((1, ph[:, None, None] * (w[:, None] * psi[to][:, :, None, :]).sum(-1)),
                          (-1, phb[:, None, None] * (_dag(w[back])[:, None] * psi[back][:, :, None, :]).sum(-1))):
            out = out + LAMBDA[n] * chi
            for mu in range(4):
                if d[mu]:
                    cols = [g[0] for g in GAMMA[mu]]
                    val = torch.tensor([g[1] for g in GAMMA[mu]], dtype=chi.dtype, device=chi.device)
                    out = out + (RHO[n] * sign * d[mu]) * val[:, None] * chi[:, cols]
    if clover is not None:
        out = out + torch.einsum("vabcd,vcd->vab", clover, psi)
    return out


def _g5(v):
    return v * torch.tensor([1.0, 1.0, -1.0, -1.0], dtype=torch.float64, device=v.device)[:, None]


def _clover(lat, U, csw):
    """-(c_SW/2) sum_{mu<nu} sigma_{mu nu} F_{mu nu}, as (V, 4, 3, 4, 3)"""
    gam = []
    for g in GAMMA:
        m = torch.zeros((4, 4), dtype=torch.complex128, device="cuda")
        for s, (col, val) in enumerate(g):
            m[s, col] = val
        gam.append(m)

    def step(at, mu, sign):
        """the link leaving each site of `at` in direction sign mu, and the sites that it reaches"""
        e = [0, 0, 0, 0]
        e[mu] = sign
        to = lat.at(e)[0][at]
        return (U[at, mu] if sign > 0 else _dag(U[to, mu])), to

    here = torch.arange(lat.V, device="cuda")
    C = 0
    for mu in range(4):
        for nu in range(mu + 1, 4):
            Q = 0
            for a, s, b, t in ((mu, 1, nu, 1), (nu, 1, mu, -1), (mu, -1, nu, -1), (nu, -1, mu, 1)):
                M, at = None, here
                for link in ((a, s), (b, t), (a, -s), (b, -t)):
                    u, at = step(at, *link)
                    M = u if M is None else _mm(M, u)
                Q = Q + M
            F = (Q - _dag(Q)) / 8j
            sigma = 0.5j * (gam[mu] @ gam[nu] - gam[nu] @ gam[mu])
            C = C - 0.5 * csw * sigma[None, :, None, :, None] * F[:, None, :, None, :]
    return C


def _solve(A, b):
    """BiCGstab, restarted from the true residual until it is at rounding level"""
    x = torch.zeros_like(b)
    dot = lambda u, v: torch.vdot(u.reshape(-1), v.reshape(-1))  # noqa: E731
    bb = dot(b, b).real
    for _ in range(4):
        r = b - A(x)
        start = dot(r, r).real
        if start <= 1e-29 * bb:
            break
        rhat, p, v = r, torch.zeros_like(r), torch.zeros_like(r)
        rho = alpha = omega = torch.ones((), dtype=b.dtype, device=b.device)
        for it in range(600):
            new = dot(rhat, r)
            p = r + (new / rho) * (alpha / omega) * (p - omega * v)
            rho = new
            v = A(p)
            alpha = rho / dot(rhat, v)
            s = r - alpha * v
            t = A(s)
            omega = dot(t, s) / dot(t, t)
            x = x + alpha * p + omega * s
            r = s - omega * t
            if it % 5 == 4 and dot(r, r).real <= max(1e-17 * start, 1e-30 * bb):
                break
    return x


def _sign(H, v):
    """sign(H) v by a Chebyshev polynomial for 1/sqrt on [0.1, 3], which holds the spectrum of H^2 for these links;
    None if applying it twice does not give v back"""
    lo, hi, N = 0.1, 3.0, 110
    j = (torch.arange(N, dtype=torch.float64) + 0.5) * math.pi / N
    f = 1 / (0.5 * (hi + lo) + 0.5 * (hi - lo) * torch.cos(j)).sqrt()
    coef = [float(2 / N * (f * torch.cos(k * j)).sum()) for k in range(N)]

    def once(v):
        T = lambda u: (2 * H(H(u)) - (hi + lo) * u) / (hi - lo)  # noqa: E731
        a, b = torch.zeros_like(v), torch.zeros_like(v)
        for k in range(N - 1, 0, -1):
            a, b = coef[k] * v + 2 * T(a) - b, a
        return H(0.5 * coef[0] * v + T(a) - b)

    s = once(v)
    return s if float((once(s) - v).norm() / v.norm()) < 1e-11 else None


def exact(c, seed):
    L, kind, n, m0 = _lattice(c), c["kind"], c.get("nrhs", 1), c["m0"]
    V = synth.volume(L)
    # longer than some twenty seconds, or more memory than the card has beside the rest
    if V > 24 ** 3 * 48 or (kind == "solve" and V * n > 16 ** 3 * 32):
        return None
    U, v = _inputs(c, seed)
    lat = _Lattice(L)
    if kind in ("dirac", "action"):
        U.requires_grad_(True)
        W = _hops(lat, U)
        with torch.no_grad():
            psi = v[0]
            if kind == "dirac":
                other, X, scale = v[1], psi, 1.0
            else:
                other = _g5(_solve(lambda u: _apply(lat, W, u, m0), _g5(psi)))  # D^dagger Z = phi
                X, scale = _solve(lambda u: _apply(lat, W, u, m0), other), -2.0
        out = _apply(lat, W, X, m0)
        dU = torch.autograd.grad((other.conj() * out).sum().real * scale, U)[0]
        with torch.no_grad():
            if kind == "dirac":
                return {"out": out.detach(), "dU": dU, "dpsi": _g5(_apply(lat, W, _g5(other), m0))}
            return {"S": (other.abs() ** 2).sum(), "dU": dU, "dphi": 2 * X}
    with torch.no_grad():
        W = _hops(lat, U)
        if kind == "build":
            order = sorted(W, key=lambda d: sum(o * 3 ** mu for mu, o in enumerate(d)))
            return torch.stack([W[d] for d in order], 1)
        clover = _clover(lat, U, c["csw"]) if c.get("csw") else None
        v = v.to(torch.complex128)
        if kind == "solve":
            return torch.stack([_solve(lambda u: _apply(lat, W, u, m0), x) for x in v])
        H = lambda u: _g5(_apply(lat, W, u, -1.0, clover))  # noqa: E731
        if kind == "overlap":
            signs = [_sign(H, x) for x in v]
            return None if any(s is None for s in signs) else torch.stack([x + _g5(s) for x, s in zip(v, signs)])
        if c["op"] == "H":
            return torch.stack([H(x) for x in v])
        if c["op"] == "Ddag":
            return torch.stack([_g5(_apply(lat, W, _g5(x), m0, clover)) for x in v])
        return torch.stack([_apply(lat, W, x, m0, clover) for x in v])

"""The work that users of this package have it do, as measured cases.

Each case names a public call (``kind``) and its sizes:

  apply      H = Gamma5 D_dwf on one or many fields (``apply_g5dwf``)
  transfer   restriction to the coarse space and prolongation back
  setup      subspace, little Dirac operator, its dense inverse, one coarse solve
  cr, cgne   the plain solvers: CR on H, red-black preconditioned CGNE
  hdcr       the two-level solve for one source
  multi      the two-level solve for the 12 spin-colour point sources at once
  grad       the differentiable solve, forward and backward

Sizes are those of the benchmark's workloads, of the tests, or generic.  Links
are exp(i eps H) with H Gaussian traceless Hermitian and eps = 0.5, the domain
wall height is 1.8.  ``exact`` restates each operation in plain torch in 64 bits.
"""
from __future__ import annotations

import math

import torch

import paper_1611_06944_gb300 as hd

M5, EPS = 1.8, 0.5
CHUNK = 6  # fields that the 64-bit restatement handles at once


def _case(kind, L, Ls, **kw):
    c = {"kind": kind, "Lx": L[0], "Ly": L[1], "Lz": L[2], "Lt": L[3], "Ls": Ls, "bc_t": 1, "mf": 0.01}
    c.update(kw)
    return c


def listed():
    return [
        # a first call on a toy lattice, and the operator of a lattice analysis on a workstation:
        # latency and launches are all there is
        _case("apply", (4, 4, 4, 4), 8, name="apply_f64_4x4x4x4_ls8", bits=64, nrhs=1, values="gauss"),
        # the operator inside every FP64 solve of the two-level workload
        _case("apply", (16, 16, 16, 16), 16, name="apply_f64_16x16x16x16_ls16", bits=64, nrhs=1, values="gauss"),
        # twelve spin-colour columns of a propagator on a lattice with odd extents
        _case("apply", (5, 7, 6, 9), 10, name="apply_f32_5x7x6x9_ls10_x12", bits=32, nrhs=12, bc_t=-1, values="wall"),
        # the FP32 operator of the mixed-precision workload, the largest lattice in use
        _case("apply", (24, 24, 24, 48), 16, name="apply_f32_24x24x24x48_ls16", bits=32, nrhs=1, mf=0.005,
              values="gauss"),
        # the coarse correction's grid transfer in the FP64 two-level workload
        _case("transfer", (16, 16, 16, 16), 16, name="transfer_f64_16x16x16x16_ls16", bits=64, nvec=24, block=4,
              nrhs=1),
        # what a new gauge configuration costs before its first solve
        _case("setup", (8, 8, 8, 16), 8, name="setup_f64_8x8x8x16_ls8", bits=64, nvec=24, block=4, order=200,
              cut=0.3),
        # plain CR, the solver that needs no setup
        _case("cr", (8, 8, 8, 8), 8, name="cr_f64_8x8x8x8_ls8", bits=64),
        # red-black preconditioned CGNE, the production solver that the method is compared with
        _case("cgne", (12, 12, 12, 12), 16, name="cgne_f64_12x12x12x12_ls16", bits=64),
        # the two-level workload's solve, all FP64
        _case("hdcr", (16, 16, 16, 16), 16, name="hdcr_f64_16x16x16x16_ls16", bits=64, nvec=24, block=4, order=200,
              cut=0.3, restart=24),
        # a light valence quark, FP32 V-cycle inside an FP64 outer iteration
        _case("hdcr", (16, 16, 16, 32), 16, name="hdcr_f32_16x16x16x32_ls16", bits=32, nvec=32, block=4, order=300,
              cut=0.2, restart=8, mf=0.001),
        # a whole propagator: twelve point sources in lockstep
        _case("multi", (8, 8, 8, 16), 8, name="multi_f32_8x8x8x16_ls8", bits=32, nvec=24, block=4, order=200,
              cut=0.3, restart=8, mf=0.05),
        # the differentiation workload in complex64
        _case("grad", (8, 8, 8, 16), 8, name="grad_f32_8x8x8x16_ls8", bits=32, nvec=16, block=4, order=100, cut=0.3,
              restart=8, mf=0.05),
    ]


def _log(rng, lo, hi):
    return lo * (hi / lo) ** rng.random()


def _extents(rng, lo, hi, most, ls, step=1):
    """Four extents, multiples of ``step``, with at most ``most`` 5d sites, spread over the logarithm."""
    while True:
        L = [max(lo, int(round(_log(rng, lo, hi) / step)) * step) for _ in range(4)]
        if L[0] * L[1] * L[2] * L[3] * ls <= most:
            return L


def draw(rng):
    kind = rng.choice(["apply"] * 5 + ["transfer", "transfer", "setup", "cr", "cgne", "hdcr", "hdcr", "multi", "grad"])
    bits = rng.choice([32, 64])
    bc = rng.choice([1, -1])
    if kind == "apply":
        ls = rng.choice([4, 6, 7, 8, 10, 12, 16, 16, 24])
        most = 10_616_832 if bits == 32 else 2_000_000
        L = _extents(rng, 3, 32, most, ls)
        sites = L[0] * L[1] * L[2] * L[3] * ls
        nrhs = max(1, min(12, int(_log(rng, 1, 13)), most // sites))
        return _case(kind, L, ls, bits=bits, nrhs=nrhs, bc_t=bc, mf=round(_log(rng, 0.001, 0.1), 5),
                     values=rng.choice(["gauss", "wall"]))
    if kind == "transfer":
        block = rng.choice([2, 3, 4])
        ls = rng.choice([6, 8, 12, 16])
        L = _extents(rng, 2 * block, 16, 1_048_576, ls, block)
        sites = L[0] * L[1] * L[2] * L[3] * ls
        nvec = rng.choice([8, 16, 20, 24, 32])
        return _case(kind, L, ls, bits=bits, nvec=nvec, block=block,
                     nrhs=max(1, min(rng.choice([1, 1, 2, 5]), 1_100_000 // sites)))
    if kind == "setup":
        ls = rng.choice([6, 8, 12])
        L = _extents(rng, 8, 16, 70_000, ls, 4)
        return _case(kind, L, ls, bits=bits, nvec=rng.choice([16, 20, 24]), block=4, order=rng.choice([100, 150, 200]),
                     cut=0.3, bc_t=bc)
    if kind == "cr":
        ls = rng.choice([6, 8, 10])
        return _case(kind, _extents(rng, 4, 12, 60_000, ls), ls, bits=64, bc_t=bc, mf=round(_log(rng, 0.01, 0.1), 4))
    if kind == "cgne":
        ls = rng.choice([7, 8, 12, 16])
        return _case(kind, _extents(rng, 4, 14, 330_000, ls, 2), ls, bits=64, bc_t=bc,
                     mf=round(_log(rng, 0.01, 0.1), 4))
    ls = rng.choice([8, 8, 12, 16])
    if kind == "hdcr":
        L = _extents(rng, 8, 16, 400_000, ls, 4)
        return _case(kind, L, ls, bits=bits, nvec=24, block=4, order=200, cut=0.3, restart=rng.choice([8, 16, 24]),
                     mf=round(_log(rng, 0.02, 0.1), 4), bc_t=bc)
    if kind == "multi":
        return _case(kind, _extents(rng, 8, 16, 70_000, 8, 4), 8, bits=bits, nvec=24, block=4, order=200, cut=0.3,
                     restart=8, mf=round(_log(rng, 0.02, 0.1), 4), bc_t=bc)
    ls = 8 if bits == 32 else rng.choice([6, 8])
    return _case(kind, _extents(rng, 8, 16, 70_000 if bits == 32 else 37_000, ls, 4), ls, bits=bits, nvec=16, block=4,
                 order=100, cut=0.3, restart=8,
                 mf=round(_log(rng, 0.05, 0.1), 4), bc_t=bc)


# ------------------------------------------------------------------ inputs
def _lat(case):
    return hd.Lattice((case["Lx"], case["Ly"], case["Lz"], case["Lt"]), case["Ls"], case["bc_t"])


def _v4(case):
    return case["Lx"] * case["Ly"] * case["Lz"] * case["Lt"]


def _dtype(case):
    return torch.complex64 if case["bits"] == 32 else torch.complex128


def _gaussian(gen, shape):
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), generator=gen, device="cuda", dtype=torch.float64))


def _links(case, gen):
    """U = exp(i eps sum_a w_a lambda_a / 2), w_a ~ N(0, 1): (4, V4, 3, 3) complex128."""
    lam = torch.zeros(8, 3, 3, dtype=torch.complex128, device="cuda")
    for a, (i, j) in enumerate(((0, 1), (0, 2), (1, 2))):
        lam[2 * a, i, j] = lam[2 * a, j, i] = 1
        lam[2 * a + 1, i, j], lam[2 * a + 1, j, i] = -1j, 1j
    lam[6] = torch.diag(torch.tensor([1, -1, 0], dtype=torch.complex128))
    lam[7] = torch.diag(torch.tensor([1, 1, -2], dtype=torch.complex128)) / math.sqrt(3.0)
    w = torch.randn((4 * _v4(case), 8), generator=gen, device="cuda", dtype=torch.float64)
    x = (1j * EPS / 2) * (w.to(torch.complex128) @ lam.reshape(8, 9)).reshape(-1, 3, 3) / 16
    term = torch.eye(3, dtype=torch.complex128, device="cuda").expand_as(x)
    U = term.clone()
    for k in range(1, 11):  # |x| < 0.2: the series of exp(x) is exact to rounding after 10 terms
        term = term @ x / k
        U = U + term
    for _ in range(4):
        U = U @ U
    return U.reshape(4, -1, 3, 3).contiguous()


def _inputs(case, seed):
    """Every input of a case, from the seed alone, at the precision that the call takes."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)
    V4, Ls, kind = _v4(case), case["Ls"], case["kind"]
    one = (V4, 12, Ls)
    d = {}
    if kind != "transfer":
        d["U"] = _links(case, gen)
    if kind in ("apply", "transfer"):
        psi = _gaussian(gen, (case["nrhs"],) + one)
        if case.get("values") == "wall":  # a quark propagator: bound to the walls, decaying into the fifth dimension
            s = torch.arange(Ls, device="cuda")
            psi = psi * torch.exp(-0.8 * torch.minimum(s, Ls - 1 - s).double())
        d["psi"] = psi.to(_dtype(case))
    elif kind == "multi":
        b = torch.zeros((12,) + one, dtype=torch.complex128, device="cuda")
        site = int(torch.randint(V4, (1,), generator=gen, device="cuda"))
        for i in range(12):
            b[i, site, i, 0] = 1.0
        d["b"] = b
    else:
        d["b"] = _gaussian(gen, one)
    if kind == "apply":
        d["U"] = d["U"].to(_dtype(case))
    if kind == "grad":
        d["U"], d["b"] = d["U"].to(_dtype(case)), d["b"].to(_dtype(case))
        d["eta"] = _gaussian(gen, one).to(_dtype(case))
    if "nvec" in case:
        n = case["nvec"] if kind == "transfer" else case["nvec"] // 2
        d["noise"] = _gaussian(gen, (n,) + one)
    if kind == "setup":
        d["c"] = _gaussian(gen, (1, V4 // case["block"] ** 4, case["nvec"])).to(torch.complex64)
    return d


def _filter_kw(case):
    # an FP32 filter shapes the subspace; the basis is stored in the precision of the V-cycle
    return dict(kind="chebyshev", order=case["order"], lam_cut=case["cut"], lam_max=8.0,
                filter_dtype=torch.complex64, store_dtype=_dtype(case))


def _two_level(case, d):
    sub = hd.build_subspace(_lat(case), d["U"], d["noise"], M5, case["mf"], (case["block"],) * 4, **_filter_kw(case))
    co = hd.build_coarse_op(sub, d["U"], M5, case["mf"], op_dtype=_dtype(case), fp32_build=case["bits"] == 64)
    hd.coarse_invert(co)
    return sub, co


def prepare(case, seed):
    state = _inputs(case, seed)
    state["case"], state["lat"] = case, _lat(case)
    if case["kind"] == "transfer":
        state["sub"] = hd.subspace_from_vectors(state["lat"], (case["block"],) * 4, state.pop("noise"),
                                                store_dtype=_dtype(case))
    elif case["kind"] in ("hdcr", "multi"):
        state["sub"], state["co"] = _two_level(case, state)
        del state["noise"]
    return state


def run(state):
    case, lat, kind = state["case"], state["lat"], state["case"]["kind"]
    if kind == "apply":
        return hd.apply_g5dwf(lat, state["U"], state["psi"], M5, case["mf"])
    if kind == "transfer":
        c = hd.restrict(state["sub"], state["psi"])
        return c, hd.prolong(state["sub"], c)
    if kind == "setup":
        sub, co = _two_level(case, state)
        return sub.vectors(), co.op(), hd.coarse_solve_dense(co, state["c"])
    if kind == "cr":
        return hd.cr_solve(lat, state["U"], state["b"], M5, case["mf"], tol=1e-10)[0]
    if kind == "cgne":
        return hd.cgne_rb_solve(lat, state["U"], state["b"], M5, case["mf"], tol=1e-10)[0]
    if kind == "hdcr":
        return hd.hdcr_solve(state["co"], state["U"], state["b"], tol=1e-10, max_outer=500, restart=case["restart"],
                             inner_dtype=_dtype(case))[0]
    if kind == "multi":
        return hd.hdcr_solve_multi(state["co"], state["U"], state["b"], tol=1e-10, max_outer=500,
                                   restart=case["restart"], inner_dtype=_dtype(case))[0]
    U, b = state["U"].detach().requires_grad_(True), state["b"].detach().requires_grad_(True)
    x = hd.solve_autograd(lat, U, b, state["noise"], M5, case["mf"], (case["block"],) * 4,
                          filter_kw=dict(kind="chebyshev", order=case["order"], lam_cut=case["cut"]),
                          solve_kw=dict(max_outer=500, restart=case["restart"]))
    torch.vdot(state["eta"].reshape(-1), x.reshape(-1)).real.backward()
    return x.detach(), U.grad, b.grad


# -------------------------------------------------------------------- work
# Applications of H that a solve cannot do without at its tolerance, as the iteration counts of the
# benchmark's workloads give them (a case's own count differs by a factor of two at most).
_APPLIES = {"cr": 1000, "cgne": 400, "hdcr": 17 * 45, "multi": 17 * 45, "grad": 2 * 17 * 45}


def work(case):
    v4, kind = _v4(case), case["kind"]
    v5 = v4 * case["Ls"]
    cb = 8 if case["bits"] == 32 else 16
    links, field = 36 * v4 * cb, 12 * v5 * cb
    if kind == "apply":
        return {"bytes": links + 2 * case["nrhs"] * field, "flops": 1416 * v5 * case["nrhs"]}
    if kind == "transfer":
        coarse = case["nvec"] * (v4 // case["block"] ** 4) * cb
        return {"bytes": (case["nvec"] + 2 * case["nrhs"]) * field + 2 * case["nrhs"] * coarse,
                "flops": 2 * 8 * case["nvec"] * 12 * v5 * case["nrhs"]}
    if kind == "setup":
        nvec, n = case["nvec"], case["nvec"] * (v4 // case["block"] ** 4)
        # the filter, one orthonormalisation, P^dag H P over the block faces and interior, the inverse
        flops = (nvec // 2 * 2 * case["order"] * 1416 * v5 + 4 * nvec * nvec * 2 * 12 * v5 + nvec * 1416 * v5
                 + 2 * 8 * nvec * nvec * 12 * v5 + 8 * n ** 3)
        return {"bytes": 36 * v4 * 16 + (nvec // 2 + nvec) * 12 * v5 * 16, "flops": flops}
    n = 12 if kind == "multi" else 1
    return {"bytes": 36 * v4 * 16 + 2 * n * 12 * v5 * 16, "flops": _APPLIES[kind] * 1416 * v5 * n}


# --------------------------------------------------------------- tolerance
def tolerance(case):
    kind, bits = case["kind"], case["bits"]
    if kind == "apply":  # measured against 64 bits: 1e-16 and 6e-8
        return {"rel": 4e-16} if bits == 64 else {"rel": 2.5e-7}
    if kind == "transfer":  # measured 9e-15 (the basis' orthonormalisation) and 2.5e-7
        return {"rel": 4e-14} if bits == 64 else {"rel": 1e-6}
    if kind == "setup":
        # measured 8e-6 (the FP32 filter, amplified where filtered vectors are nearly parallel) and 6e-5 (the FP32 inverse)
        return {"rel": 2.5e-4}
    if kind == "grad":  # measured 6e-6 in FP32 (the solve's tolerance is 1e-7); 1e-10 in FP64
        return {"rel": 2.5e-5} if bits == 32 else {"rel": 1e-7}
    # solves to a residual of 1e-10: solutions of two solvers differ by up to 2e-8 on the lightest quark
    return {"rel": 8e-8, "max": 1e-5}


# ------------------------------------------------------------------- exact
def _isigma(k, v):
    """i sigma_k on the spin axis (-3) of (..., 2, 3, Ls)."""
    a, b = v[..., 0, :, :], v[..., 1, :, :]
    if k == 0:
        return torch.stack((1j * b, 1j * a), -3)
    if k == 1:
        return torch.stack((b, -a), -3)
    return torch.stack((1j * a, -1j * b), -3)


class _Operator:
    """H = Gamma5 D_dwf on (n, V4, 12, Ls) complex128 fields, in plain torch."""

    def __init__(self, case, U):
        self.case = case
        self.shape = (case["Lt"], case["Lz"], case["Ly"], case["Lx"])
        self.U = U.to(torch.complex128).reshape((4,) + self.shape + (3, 3))

    def _shift(self, v, mu, sign):
        """v(x + sign mu), with the boundary phase in t; v has the lattice on axes 1..4."""
        out = torch.roll(v, -sign, dims=4 - mu)
        if mu == 3 and self.case["bc_t"] != 1:
            out[:, -1 if sign > 0 else 0] *= self.case["bc_t"]
        return out

    def hop(self, psi, mu, sign, U=None):
        """(1 -+ gamma_mu) U psi(x +- mu) of (n, Lt, Lz, Ly, Lx, 4, 3, Ls) fields."""
        U = self.U if U is None else U
        up, dn = psi[..., :2, :, :], psi[..., 2:, :, :]
        t = dn if mu == 3 else _isigma(mu, dn)
        # (1 - gamma_k) keeps u + i sigma_k d, (1 - gamma_t) keeps u - d
        h = up + t if (sign > 0) == (mu < 3) else up - t
        if sign > 0:
            h = torch.matmul(U[mu].unsqueeze(-3), self._shift(h, mu, 1))
        else:
            h = self._shift(torch.matmul(U[mu].mH.unsqueeze(-3), h), mu, -1)
        low = h if mu == 3 else _isigma(mu, h)
        return torch.cat((h, -low if sign > 0 else low), -3)

    def local(self, psi):
        mf = self.case["mf"]
        out = (5.0 - M5) * psi
        nxt, prv = torch.roll(psi, -1, dims=-1), torch.roll(psi, 1, dims=-1)
        nxt[..., -1] *= -mf
        prv[..., 0] *= -mf
        out[..., 2:, :, :] -= nxt[..., 2:, :, :]
        out[..., :2, :, :] -= prv[..., :2, :, :]
        return out

    @staticmethod
    def gamma5_r5(v):
        out = torch.flip(v, dims=(-1,))
        out[..., 2:, :, :] *= -1
        return out

    def fields(self, v):
        return v.reshape((-1,) + self.shape + (4, 3, self.case["Ls"]))

    def __call__(self, v, U=None):
        psi = self.fields(v)
        out = self.local(psi)
        for mu in range(4):
            for sign in (1, -1):
                out = out - 0.5 * self.hop(psi, mu, sign, U)
        return self.gamma5_r5(out).reshape(v.shape)

    def chunked(self, v):
        return torch.cat([self(v[i:i + CHUNK]) for i in range(0, v.shape[0], CHUNK)])


def _dots(a, b):
    return (a.conj() * b).real.flatten(1).sum(1).reshape(-1, 1, 1, 1)


def _solve(H, b):
    """H x = b for each field of b: conjugate gradients on H^2, started again once from the true residual."""
    x = torch.zeros_like(b)
    for _ in range(2):
        r = H(b - H(x))
        p, rr = r.clone(), _dots(r, r)
        stop, dx = rr * 1e-20, torch.zeros_like(b)
        for _ in range(200):
            for _ in range(25):
                hp = H(p)
                a = rr / _dots(hp, hp).clamp_min(1e-300)
                dx += a * p
                r = r - a * H(hp)
                new = _dots(r, r)
                p = r + (new / rr.clamp_min(1e-300)) * p
                rr = new
            if bool((rr <= stop).all()):
                break
        x = x + dx
    return x


def _blocks(case, v):
    """(n, V4, 12, Ls) -> (n, Vc, K), the sites of a block together."""
    B, n = case["block"], v.shape[0]
    Lc = [case[k] // B for k in ("Lt", "Lz", "Ly", "Lx")]
    a = v.reshape(n, Lc[0], B, Lc[1], B, Lc[2], B, Lc[3], B, 12 * case["Ls"])
    return a.permute(0, 1, 3, 5, 7, 2, 4, 6, 8, 9).reshape(n, Lc[0] * Lc[1] * Lc[2] * Lc[3], -1)


def _unblocks(case, w):
    B, n = case["block"], w.shape[0]
    Lc = [case[k] // B for k in ("Lt", "Lz", "Ly", "Lx")]
    a = w.reshape(n, *Lc, B, B, B, B, 12 * case["Ls"]).permute(0, 1, 5, 2, 6, 3, 7, 4, 8, 9)
    return a.reshape(n, _v4(case), 12, case["Ls"])


def _orthonormal(phi):
    """(nvec, Vc, K) block vectors orthonormalised in order: three rounds of Cholesky QR."""
    for _ in range(3):
        V = phi.permute(1, 2, 0)
        R = torch.linalg.cholesky(V.mH @ V).mH
        phi = torch.linalg.solve_triangular(R, V, upper=True, left=False).permute(2, 0, 1)
    return phi.contiguous()


def _filtered(case, H, x):
    lo, hi = case["cut"] ** 2, 64.0
    a, b = 2.0 / (hi - lo), -(hi + lo) / (hi - lo)

    def t(v):
        return a * H.chunked(H.chunked(v)) + b * v
    prev, cur = x, t(x)
    for k in range(2, case["order"] + 1):
        prev, cur = cur, 2.0 * t(cur) - prev
        if k % 8 == 0:
            s = 1.0 / torch.linalg.vector_norm(cur)
            prev, cur = prev * s, cur * s
    return cur


def _little(case, H, phi):
    """(Vc, 9, nvec, nvec): <phi_j^a | H | phi_k^(a + leg)>, the self leg without the hops that leave the block."""
    fields = _unblocks(case, phi)
    nvec, Vc = phi.shape[0], phi.shape[1]
    A = torch.zeros(Vc, 9, nvec, nvec, dtype=torch.complex128, device="cuda")
    bra = phi.permute(1, 0, 2).conj()

    def project(y):
        return bra @ _blocks(case, y).permute(1, 2, 0)

    own = H.chunked(fields)
    grid = torch.meshgrid(*[torch.arange(n, device="cuda") for n in H.shape], indexing="ij")
    for mu in range(4):
        for sign in (1, -1):
            edge = grid[3 - mu] % case["block"] == (case["block"] - 1 if sign > 0 else 0)
            out = []
            for i in range(0, nvec, CHUNK):
                psi = H.fields(fields[i:i + CHUNK])
                y = H.gamma5_r5(-0.5 * H.hop(psi, mu, sign)) * edge.reshape((1,) + H.shape + (1, 1, 1))
                out.append(y.reshape(fields[i:i + CHUNK].shape))
            y = torch.cat(out)
            own -= y
            A[:, 1 + 2 * mu + (0 if sign > 0 else 1)] = project(y)
    A[:, 0] = project(own)
    return A


def _dense(case, A):
    Vc, nvec = A.shape[0], A.shape[-1]
    Lc = [case[k] // case["block"] for k in ("Lt", "Lz", "Ly", "Lx")]
    idx = torch.arange(Vc, device="cuda").reshape(Lc)
    D = torch.zeros(Vc, nvec, Vc, nvec, dtype=torch.complex128, device="cuda")
    a = idx.reshape(-1)
    for leg in range(9):
        mu, sign = (leg - 1) // 2, 1 if leg % 2 else -1
        nb = a if leg == 0 else torch.roll(idx, -sign, dims=3 - mu).reshape(-1)
        D[a, :, nb, :] += A[:, leg]
    return D.reshape(Vc * nvec, Vc * nvec)


def exact(case, seed):
    kind = case["kind"]
    v5 = _v4(case) * case["Ls"]
    if kind in ("cr", "cgne", "hdcr", "grad") and v5 > 140_000 or kind == "multi" and v5 > 70_000:
        return None  # the 64-bit restatement of such a solve takes minutes
    d = _inputs(case, seed)
    if kind == "transfer":
        phi = _orthonormal(_blocks(case, d["noise"]))
        psi = _blocks(case, d["psi"].to(torch.complex128))
        c = torch.einsum("jak,nak->naj", phi.conj(), psi)
        return c, _unblocks(case, torch.einsum("jak,naj->nak", phi, c))
    H = _Operator(case, d["U"])
    if kind == "apply":
        return torch.cat([H(p.to(torch.complex128)[None]) for p in d["psi"]])
    if kind == "setup":
        x = _filtered(case, H, d["noise"])
        g = H.gamma5_r5(H.fields(x)).reshape(x.shape)
        phi = _orthonormal(_blocks(case, torch.cat((0.5 * (x + g), 0.5 * (x - g)))))
        A = _little(case, H, phi)
        c = torch.linalg.solve(_dense(case, A), d["c"].to(torch.complex128).reshape(-1))
        return _unblocks(case, phi), A, c.reshape(d["c"].shape)
    if kind != "grad":
        b = d["b"] if kind == "multi" else d["b"][None]
        return _solve(H, b).reshape(d["b"].shape)
    b, eta = d["b"].to(torch.complex128), d["eta"].to(torch.complex128)
    x, y = _solve(H, torch.stack((b, eta)))
    U = H.U.detach().requires_grad_(True)
    # d Re(eta^dag x) = -Re(y^dag dH x), y = H^-1 eta
    (-torch.vdot(y.reshape(-1), H(x[None], U).reshape(-1)).real).backward()
    return x, U.grad.reshape(4, -1, 3, 3), y

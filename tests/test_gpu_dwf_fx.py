"""The FP64 operator in fixed point (dwf_fx.cu): its error against extended precision, every
form a call can take (scratch for all fields, for one, for none), operands outside the
format, and the fused epilogues of the solver against the oracle's V-cycle."""
import ctypes

import numpy as np
import pytest

import synth
from oracle import dwf, multigrid as mg
from gpu_util import dev, host, links, natural, planes, relerr

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def hd():
    import paper_1611_06944_gb300 as hd
    return hd


def apply_with(hd, lat, U, psi, scratch_fields, mf=0.01):
    """H psi through the C entry with scratch for that many fields (0: the FP64 kernel)."""
    g, p = lat.c_geom(), hd._params(1.8, mf)
    n = psi.numel() // (12 * lat.V5)
    size = hd._L.hdcr_apply_scratch_bytes(hd.C_ref(g), 0, scratch_fields) if scratch_fields else 0
    scratch = torch.empty(size, dtype=torch.uint8, device="cuda")
    out = torch.empty_like(psi)
    s = hd._L.hdcr_apply_g5dwf_scratch(hd.C_ref(g), hd.C_ref(p), U.data_ptr(), psi.data_ptr(), out.data_ptr(), 0, n,
                                       scratch.data_ptr() if size else None, size,
                                       ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert s == 0
    return out


def apply_extended(U, psi, mf, bc):
    """dwf.apply_H in extended precision (numpy longdouble), its pieces rewritten without BLAS."""
    U, p = U.astype(np.clongdouble), psi.astype(np.clongdouble)
    G = [g.astype(np.clongdouble) for g in dwf.GAMMA]
    one = np.eye(4, dtype=np.clongdouble)

    def colour(M, v):
        return (M[..., None, None, :, :] * v[..., None, :]).sum(-1)

    def spin(S, v):
        return (S[:, :, None] * v[..., None, :, :]).sum(-2)

    D = np.longdouble(5.0 - 1.8) * p
    nxt, prv = np.roll(p, -1, -3), np.roll(p, 1, -3)
    nxt[..., -1, :, :] *= -np.longdouble(mf)
    prv[..., 0, :, :] *= -np.longdouble(mf)
    D[..., 2:, :] -= nxt[..., 2:, :]
    D[..., :2, :] -= prv[..., :2, :]
    for mu in range(4):
        fwd = spin(one - G[mu], colour(U[mu], dwf.shift_fermion(p, mu, +1, bc)))
        dag = np.conj(np.swapaxes(dwf.shift_links(U[mu], mu, -1), -1, -2))
        bwd = spin(one + G[mu], colour(dag, dwf.shift_fermion(p, mu, -1, bc)))
        D = D - np.longdouble(0.5) * (fwd + bwd)
    out = D[..., ::-1, :, :].copy()
    out[..., 2:, :] *= -1
    return out


# tiles that divide the lattice and that do not, partial warps, Ls from 2 to the largest a
# tile takes (256) and one beyond it (the FP64 kernel)
SHAPES = [((4, 4, 4, 4), 8, 1), ((3, 5, 2, 6), 5, -1), ((7, 3, 5, 2), 16, 1), ((4, 2, 2, 4), 2, -1),
          ((5, 3, 1, 7), 3, 1), ((2, 2, 3, 2), 33, -1), ((2, 1, 2, 2), 256, 1), ((2, 1, 2, 2), 258, -1)]


@pytest.mark.parametrize("L,Ls,bc", SHAPES)
@pytest.mark.parametrize("wall", [False, True])
def test_error_is_not_above_the_fp64_kernels(hd, L, Ls, bc, wall):
    U = synth.gauge_field(L, 0.5, 5000)
    psi = synth.gaussian_fermion(L, Ls, 5001, count=3)
    if wall:  # decaying into the fifth dimension
        s = np.arange(Ls)
        psi = psi * np.exp(-0.5 * np.minimum(s, Ls - 1 - s))[:, None, None]
    lat = hd.Lattice(L, Ls, bc)
    Ud, pd = dev(links(U)), dev(planes(psi))
    want = np.stack([apply_extended(U, p, 0.01, bc) for p in psi])

    def err(t):
        d = natural(host(t), L, Ls) - want
        return float(np.sqrt((np.abs(d) ** 2).sum() / (np.abs(want) ** 2).sum()))

    fp64 = err(apply_with(hd, lat, Ud, pd, 0))
    full = hd.apply_g5dwf(lat, Ud, pd, 1.8, 0.01)
    # 5e-17 measured on every shape, 1.5e-16 for the FP64 kernel
    assert err(full) <= fp64 <= 2.5e-16
    for k in (3, 2, 1):
        assert torch.equal(apply_with(hd, lat, Ud, pd, k), full)


@pytest.mark.parametrize("value", [float("nan"), float("inf"), 1e200, 1e-250, 5e-324, 0.0])
def test_operands_outside_the_format(hd, value):
    """A site that holds such a value (one component, or a whole site of it) and a link that is
    not finite: finite results as the FP64 kernel's, infinities and NaN where it has them."""
    L, Ls, bc = (4, 3, 2, 4), 6, -1
    lat = hd.Lattice(L, Ls, bc)
    U0 = dev(links(synth.gauge_field(L, 0.5, 5100)))
    p0 = dev(planes(synth.gaussian_fermion(L, Ls, 5101)))
    for what in ("component", "site", "link", "all"):
        U, psi = U0.clone(), p0.clone()
        if what == "component":
            psi[5, 3, 2] = value
        elif what == "site":
            psi[5, :, 2] = value
        elif what == "all":
            psi[:] = value
        else:
            U[1, 7, 0, 1] = value
        a = torch.view_as_real(apply_with(hd, lat, U, psi, 1))
        b = torch.view_as_real(apply_with(hd, lat, U, psi, 0))
        assert torch.equal(torch.isnan(a), torch.isnan(b))
        assert torch.equal(torch.isposinf(a), torch.isposinf(b)) and torch.equal(torch.isneginf(a), torch.isneginf(b))
        f = torch.isfinite(b)
        # per element against the sum of the magnitudes of what a site adds up (24 terms of |psi| <= 10 where
        # no large value is read): a site next to 1e200 only to its own scale
        scale = b.abs().masked_fill(~f, 0).reshape(lat.V4, 12, Ls, 2).amax(dim=(1, 3), keepdim=True).expand(
            lat.V4, 12, Ls, 2).reshape(b.shape).clamp_min(1.0 if what != "all" else 0.0)
        assert bool(((a - b).abs()[f] <= 4e-15 * scale[f] + 1e-322).all())


def test_coefficients_outside_the_format(hd):
    L, Ls = (2, 3, 2, 2), 4
    lat = hd.Lattice(L, Ls)
    U = dev(links(synth.gauge_field(L, 0.5, 5200)))
    psi = dev(planes(synth.gaussian_fermion(L, Ls, 5201)))
    for mf in (0.0, 1.0, 1e-60, 1e60):
        a, b = apply_with(hd, lat, U, psi, 1, mf), apply_with(hd, lat, U, psi, 0, mf)
        assert relerr(host(a), host(b)) <= 4e-16


@pytest.mark.parametrize("cycle", ["symmetric", "post"])
@pytest.mark.parametrize("order", [1, 2, 3])
def test_short_smoothers_match_the_oracle(hd, order, cycle):
    """One outer iteration with smoothers whose recurrence ends in its first, second and third
    step: each has an epilogue of its own."""
    L, Ls, block, M5, mf = (4, 4, 4, 4), 6, (2, 2, 2, 2), 1.8, 0.05
    U = synth.gauge_field(L, 0.3, 5300)
    b = synth.gaussian_fermion(L, Ls, 5301)
    vec = synth.gaussian_fermion(L, Ls, 5302, count=8)
    lat = hd.Lattice(L, Ls)
    Ud, bd = dev(links(U)), dev(planes(b))
    sub = hd.subspace_from_vectors(lat, block, dev(planes(vec)))
    co = hd.build_coarse_op(sub, Ud, M5, mf)
    x = torch.zeros_like(bd)
    hd.hdcr_solve_into(co, Ud, bd, x, tol=1e-14, max_outer=1, restart=1, smoother_order=order, coarse_solver="cr",
                       coarse_tol=1e-13, coarse_max=20000, cycle=cycle)
    p = mg.HDCRParams(M5=M5, mf=mf, bc_t=1)
    osub = mg.basis_from_vectors(mg.Geometry(L, Ls, block), vec)
    A = mg.coarse_op(U, osub, M5, mf, 1)
    D = mg.coarse_dense(A, osub.geom)

    def S(r):
        return mg.chebyshev_smoother(U, r, p, 1.0, 64.0, order)

    def Q(c):
        return np.linalg.solve(D, c.reshape(-1)).reshape(c.shape)

    z = mg.vcycle(U, osub, A, b, p, S=S, Qc=Q, cycle=cycle)
    w = dwf.apply_H(U, z, M5, mf, 1)
    want = np.vdot(w, b) / np.vdot(w, w).real * z
    # the coarse solve's tolerance over the smallest coarse eigenvalue bounds the difference
    assert relerr(natural(host(x), L, Ls), want) <= 1e-9


@pytest.mark.parametrize("L,Ls,bc", [((4, 6, 2, 8), 7, -1), ((2, 2, 4, 2), 33, 1), ((6, 4, 2, 2), 2, -1)])
def test_red_black_shapes(hd, L, Ls, bc):
    """CGNE's fixed-point hops on half lattices whose boxes do not fill a tile, odd and long Ls."""
    U, b, mf = synth.gauge_field(L, 0.4, 5400), synth.gaussian_fermion(L, Ls, 5401), 0.1
    x, st = hd.cgne_rb_solve(hd.Lattice(L, Ls, bc), dev(links(U)), dev(planes(b)), 1.8, mf, tol=1e-10)
    r = b - dwf.apply_H(U, natural(host(x), L, Ls), 1.8, mf, bc)
    # the Schur residual stops at 1e-10; the reconstruction adds rounding times the condition number
    assert np.linalg.norm(r) <= 2e-10 * np.linalg.norm(b)


@pytest.mark.parametrize("order", [1, 2, 16, 17, 40])
def test_fp64_filter_matches_the_oracle(hd, order):
    """The FP64 Chebyshev filter's encoded steps around its rescalings, three fields at once, on a
    basis that one orthonormalisation of the oracle's filtered vectors must reproduce."""
    L, Ls, block, mf = (4, 4, 2, 4), 5, (2, 2, 1, 2), 0.05
    U = synth.gauge_field(L, 0.4, 5500)
    noise = synth.gaussian_fermion(L, Ls, 5501, count=3)
    sub = hd.build_subspace(hd.Lattice(L, Ls), dev(links(U)), dev(planes(noise)), 1.8, mf, block, order=order,
                            lam_cut=0.5)
    g = mg.Geometry(L, Ls, block)
    f = np.stack([mg.chebyshev_filter(U, n, 1.8, mf, 1, 0.5, 8.0, order) for n in noise])
    phi = mg.block_orthonormalise(mg.to_blocks(g, mg.chiral_split(f)))
    want = np.stack([mg.from_blocks(g, v) for v in phi])
    # order x 1e-16 of rounding a step times the blocks' condition number
    assert relerr(natural(host(sub.vectors()), L, Ls), want) <= 1e-10


@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_filter_with_modes_far_above_its_interval(hd, dtype):
    """lam_max at 0.35 of the spectrum's top: modes at t = 15, which grow by 30 a step, must not
    take the recurrence or the rescaling's norm out of range."""
    L, Ls, block, mf = (4, 4, 2, 4), 5, (2, 2, 1, 2), 0.05
    U = synth.gauge_field(L, 0.4, 5500)
    noise = synth.gaussian_fermion(L, Ls, 5501, count=2)
    sub = hd.build_subspace(hd.Lattice(L, Ls), dev(links(U)), dev(planes(noise)), 1.8, mf, block, order=24,
                            lam_cut=0.5, lam_max=2.5, filter_dtype=torch.complex64 if dtype == "c64" else torch.complex128)
    g = mg.Geometry(L, Ls, block)
    f = np.stack([mg.chebyshev_filter(U, n, 1.8, mf, 1, 0.5, 2.5, 24) for n in noise])
    phi = mg.block_orthonormalise(mg.to_blocks(g, mg.chiral_split(f)))
    want = np.stack([mg.from_blocks(g, v) for v in phi])
    # the blocks' vectors have a condition number of 2.2; 24 steps of about 10 roundings each
    assert relerr(natural(host(sub.vectors()), L, Ls), want) <= (1e-4 if dtype == "c64" else 1e-11)


def links_of(kind, L):
    U = synth.gauge_field(L, 0.5, 5600)
    if kind == "random":
        return U
    one = np.zeros_like(U)
    phase = np.random.default_rng(5601).uniform(-np.pi, np.pi, U.shape[:-2] + (2,))
    for c, t in enumerate((phase[..., 0], phase[..., 1], -phase[..., 0] - phase[..., 1])):
        one[..., c, c] = np.exp(1j * t) if kind == "diagonal" else 1.0
    return one


@pytest.mark.parametrize("link", ["unit", "diagonal", "random"])
@pytest.mark.parametrize("grade", ["colour", "colour_near", "spin", "imaginary", "spread", "zeros"])
def test_components_of_different_size(hd, link, grade):
    """Components of a site of very different sizes, with links that mix them and that do not: the error of
    each component, relative to that component, is not above the FP64 kernel's."""
    L, Ls, bc = (4, 6, 4, 4), 6, -1
    U = links_of(link, L)
    psi = synth.gaussian_fermion(L, Ls, 5602)
    rng = np.random.default_rng(5603)
    if grade == "colour":
        psi = psi * np.array([1.0, 1e-5, 1e-10])
    elif grade == "colour_near":
        psi = psi * np.array([1.0, 0.1, 0.02])
    elif grade == "spin":
        psi = psi * np.array([1.0, 1e-3, 1e-6, 1e-9])[:, None]
    elif grade == "imaginary":
        psi = psi.real + 1e-9j * psi.imag
    elif grade == "spread":
        psi = psi * 2.0 ** rng.uniform(-45.0, 0.0, psi.shape)
    else:
        psi = psi * rng.integers(0, 2, psi.shape)
    lat = hd.Lattice(L, Ls, bc)
    Ud, pd = dev(links(U)), dev(planes(psi))
    want = apply_extended(U, psi, 0.01, bc)
    fx = natural(host(hd.apply_g5dwf(lat, Ud, pd, 1.8, 0.01)), L, Ls)
    fp64 = natural(host(apply_with(hd, lat, Ud, pd, 0)), L, Ls)
    for part in (np.real, np.imag):
        # per (spin, colour), and per site over all of them against the site's own terms
        e, f, w = (np.sqrt((part(a).reshape(-1, 12).astype(np.longdouble) ** 2).sum(0)) for a in (fx - want, fp64 - want, want))
        # FP64: about 2e-16 of a component (a few of its roundings); both are sums of 2304 random roundings each
        assert (e <= 1.15 * f + 1e-17 * w).all(), (part.__name__, e / w, f / w)


def one_colour(a):
    a = a.copy()
    a[..., 1:] = 0.0
    return a


@pytest.mark.parametrize("cycle", ["symmetric", "post"])
@pytest.mark.parametrize("order", [1, 2, 3])
def test_short_smoothers_where_every_site_is_computed_in_fp64(hd, order, cycle):
    """As above with links that do not mix the colours and fields of one colour, whose zero components
    no sum can make certain: each epilogue behind the FP64 arithmetic, from the FP64 operands that
    the solver keeps beside the encoded ones."""
    L, Ls, block, M5, mf = (4, 4, 4, 4), 6, (2, 2, 2, 2), 1.8, 0.05
    U = links_of("diagonal", L)
    b = one_colour(synth.gaussian_fermion(L, Ls, 5701))
    vec = one_colour(synth.gaussian_fermion(L, Ls, 5702, count=8))
    lat = hd.Lattice(L, Ls)
    Ud, bd = dev(links(U)), dev(planes(b))
    sub = hd.subspace_from_vectors(lat, block, dev(planes(vec)))
    co = hd.build_coarse_op(sub, Ud, M5, mf)
    x = torch.zeros_like(bd)
    hd.hdcr_solve_into(co, Ud, bd, x, tol=1e-14, max_outer=1, restart=1, smoother_order=order, coarse_solver="cr",
                       coarse_tol=1e-13, coarse_max=20000, cycle=cycle)
    p = mg.HDCRParams(M5=M5, mf=mf, bc_t=1)
    osub = mg.basis_from_vectors(mg.Geometry(L, Ls, block), vec)
    A = mg.coarse_op(U, osub, M5, mf, 1)
    D = mg.coarse_dense(A, osub.geom)

    def S(r):
        return mg.chebyshev_smoother(U, r, p, 1.0, 64.0, order)

    def Q(c):
        return np.linalg.solve(D, c.reshape(-1)).reshape(c.shape)

    z = mg.vcycle(U, osub, A, b, p, S=S, Qc=Q, cycle=cycle)
    w = dwf.apply_H(U, z, M5, mf, 1)
    want = np.vdot(w, b) / np.vdot(w, w).real * z
    assert relerr(natural(host(x), L, Ls), want) <= 1e-9


@pytest.mark.parametrize("solver", ["cr", "cgne", "hdcr", "multi"])
def test_solvers_where_every_site_is_computed_in_fp64(hd, solver):
    L, Ls, block, M5, mf, bc = (4, 4, 4, 4), 6, (2, 2, 2, 2), 1.8, 0.1, -1
    U = links_of("diagonal", L)
    b = one_colour(synth.gaussian_fermion(L, Ls, 5801, count=3))
    lat = hd.Lattice(L, Ls, bc)
    Ud, bd = dev(links(U)), dev(planes(b))
    if solver in ("hdcr", "multi"):
        vec = one_colour(synth.gaussian_fermion(L, Ls, 5802, count=8))
        co = hd.build_coarse_op(hd.subspace_from_vectors(lat, block, dev(planes(vec))), Ud, M5, mf)
        hd.coarse_invert(co)
    if solver == "multi":
        x = hd.hdcr_solve_multi(co, Ud, bd, tol=1e-10, max_outer=300, restart=8, inner_dtype=torch.complex128)[0]
    else:
        solve = {"cr": lambda v: hd.cr_solve(lat, Ud, v, M5, mf, tol=1e-10), "cgne": lambda v: hd.cgne_rb_solve(
            lat, Ud, v, M5, mf, tol=1e-10), "hdcr": lambda v: hd.hdcr_solve(co, Ud, v, tol=1e-10, max_outer=300, restart=8,
                                                                           inner_dtype=torch.complex128)}[solver]
        x = torch.stack([solve(v.contiguous())[0] for v in bd.reshape(3, -1, *bd.shape[-2:])])
    for f, s in zip(natural(host(x), L, Ls).reshape((3,) + b.shape[1:]), b):
        r = s - dwf.apply_H(U, f, M5, mf, bc)
        # the recursive (Schur) residual stops at 1e-10; rounding times the condition number beside it
        assert np.linalg.norm(r) <= 2e-10 * np.linalg.norm(s)
        assert not f[..., 1:].any()


def test_filter_where_every_site_is_computed_in_fp64(hd):
    """The FP64 filter on fields whose colours are graded by 1e-5 and 1e-10 with links that do not mix them:
    one noise field, whose two chiral halves are only normalised in each block."""
    L, Ls, block, mf, order = (4, 4, 2, 4), 5, (4, 4, 2, 4), 0.05, 20
    U = links_of("diagonal", L)
    noise = synth.gaussian_fermion(L, Ls, 5901, count=1) * np.array([1.0, 1e-5, 1e-10])
    block = (2, 2, 1, 2)
    sub = hd.build_subspace(hd.Lattice(L, Ls), dev(links(U)), dev(planes(noise)), 1.8, mf, block, order=order,
                            lam_cut=0.5)
    g = mg.Geometry(L, Ls, block)
    f = np.stack([mg.chebyshev_filter(U, n, 1.8, mf, 1, 0.5, 8.0, order) for n in noise])
    phi = mg.block_orthonormalise(mg.to_blocks(g, mg.chiral_split(f)))
    want = np.stack([mg.from_blocks(g, v) for v in phi])
    got = natural(host(sub.vectors()), L, Ls)
    for c in range(3):  # each colour on its own scale; 20 steps of rounding
        assert relerr(got[..., c], want[..., c]) <= 1e-12


def test_c_entry_allocates_nothing(hd):
    """hdcr_apply_g5dwf in FP64 takes no memory from the device's pool, eagerly and captured (an
    allocation node would keep a graph from running twice at once), and is the FP64 kernel."""
    L, Ls = (4, 4, 2, 4), 6
    lat = hd.Lattice(L, Ls)
    U = dev(links(synth.gauge_field(L, 0.5, 6000)))
    psi = dev(planes(synth.gaussian_fermion(L, Ls, 6001, count=2)))
    g, p = lat.c_geom(), hd._params(1.8, 0.01)
    hd._L.hdcr_apply_scratch_bytes
    with open("/proc/self/maps") as f:
        path = next(line.split()[-1] for line in f if "libcudart" in line)
    rt = ctypes.CDLL(path)
    pool, used, zero = ctypes.c_void_p(), ctypes.c_uint64(), ctypes.c_uint64(0)
    assert rt.cudaDeviceGetDefaultMemPool(ctypes.byref(pool), torch.cuda.current_device()) == 0
    used_high = 8  # cudaMemPoolAttrUsedMemHigh

    def call(out):
        assert hd._L.hdcr_apply_g5dwf(hd.C_ref(g), hd.C_ref(p), U.data_ptr(), psi.data_ptr(), out.data_ptr(), 0, 2,
                                      ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0

    want = apply_with(hd, lat, U, psi, 0)
    eager, captured, binding = torch.empty_like(psi), torch.zeros_like(psi), torch.zeros_like(psi)
    torch.cuda.synchronize()
    assert rt.cudaMemPoolSetAttribute(pool, used_high, ctypes.byref(zero)) == 0
    call(eager)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(captured)
        hd.apply_g5dwf(lat, U, psi, 1.8, 0.01, out=binding)
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    assert rt.cudaMemPoolGetAttribute(pool, used_high, ctypes.byref(used)) == 0
    assert used.value == 0
    assert torch.equal(eager, want) and torch.equal(captured, want) and torch.equal(binding, want)


@pytest.mark.parametrize("L,Ls,n", [((3, 3, 3, 2), 7, 3), ((3, 5, 3, 3), 7, 6), ((5, 3, 1, 3), 2, 12), ((4, 4, 2, 2), 4, 5)])
def test_binding_asks_for_scratch_of_all_fields(hd, L, Ls, n):
    """V5 = 2, 1, 2 and 0 mod 4: the exponents of n fields are rounded up once, not n times.  One encoding
    and one operator launch."""
    lat = hd.Lattice(L, Ls)
    U = dev(links(synth.gauge_field(L, 0.5, 6100)))
    psi = dev(planes(synth.gaussian_fermion(L, Ls, 6101, count=n)))
    before = hd._L.hdcr_launch_count()
    out = hd.apply_g5dwf(lat, U, psi, 1.8, 0.01)
    assert hd._L.hdcr_launch_count() - before == 2
    assert torch.equal(out, apply_with(hd, lat, U, psi, n))

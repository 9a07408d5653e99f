"""Restriction and prolongation (FP64 in fixed point, FP32 with several fields a pass): error
against extended precision over block shapes, vector
counts, numbers of fields, odd and even Ls and field profiles, and FP64 values outside the format."""
import numpy as np
import pytest

import synth
from gpu_util import dev, host, planes

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def hd():
    import paper_1611_06944_gb300 as hd
    return hd


def blocks(a, L, Ls, block):
    """(n, V4, 12, Ls) -> (n, Vc, K)"""
    n = a.shape[0]
    B = tuple(block[::-1])
    T = tuple(L[::-1])
    a = a.reshape((n,) + tuple(v for mu in range(4) for v in (T[mu] // B[mu], B[mu])) + (12 * Ls,))
    return a.transpose(0, 1, 3, 5, 7, 2, 4, 6, 8, 9).reshape(n, -1, int(np.prod(B)) * 12 * Ls)


# blocks of less than a round of a CTA's threads, not a multiple of them, and many rounds; clusters of
# 1, 2 and 8 CTAs; vector counts around the 8 of a CTA; numbers of fields around the 4 of a pass
CASES = [((4, 4, 4, 4), 6, (2, 2, 2, 2), 2, 1, True), ((6, 3, 9, 6), 5, (3, 1, 3, 3), 8, 2, False),
         ((8, 4, 4, 4), 16, (4, 2, 2, 2), 10, 1, True), ((8, 8, 8, 8), 8, (4, 4, 4, 4), 34, 1, False),
         ((4, 4, 4, 4), 24, (2, 2, 2, 2), 18, 5, True), ((4, 4, 4, 4), 7, (2, 2, 2, 2), 6, 4, False)]


@pytest.mark.parametrize("L,Ls,block,nvec,nrhs,wall", CASES)
@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_transfer_error(hd, L, Ls, block, nvec, nrhs, wall, dtype):
    td = torch.complex128 if dtype == "c128" else torch.complex64
    vec = synth.gaussian_fermion(L, Ls, 6000, count=nvec)
    v = synth.gaussian_fermion(L, Ls, 6001, count=nrhs)
    if wall:
        s = np.arange(Ls)
        w = np.exp(-0.5 * np.minimum(s, Ls - 1 - s))[:, None, None]
        vec, v = vec * w, v * w
    lat = hd.Lattice(L, Ls)
    sub = hd.subspace_from_vectors(lat, block, dev(planes(vec)), store_dtype=td)
    vd = dev(planes(v)).to(td)
    c = hd.restrict(sub, vd)
    f = hd.prolong(sub, c)
    phi = blocks(host(sub.vectors()), L, Ls, block).astype(np.clongdouble)
    vb = blocks(host(vd), L, Ls, block).astype(np.clongdouble)
    want = np.stack([(np.conj(phi) * x).sum(-1).T for x in vb])            # (nrhs, Vc, nvec)
    got = host(c).astype(np.clongdouble)

    def rel(a, b):
        return float(np.sqrt((np.abs(a - b) ** 2).sum() / (np.abs(b) ** 2).sum()))

    # FP64: sites summed exactly and rounded to u = 1.1e-16, a few tens of them a thread added in FP64,
    # over sums that cancel to 1 / sqrt(n) of their terms; FP32: up to 400 products a thread
    bound = 4e-16 if dtype == "c128" else 2e-6
    assert rel(got, want) <= bound
    wf = np.stack([(phi * x.T[:, :, None]).sum(0) for x in got])
    assert rel(blocks(host(f), L, Ls, block), wf) <= bound


@pytest.mark.parametrize("value", [float("nan"), float("inf"), 1e250, 1e-250, 0.0])
def test_values_outside_the_format(hd, value):
    L, Ls, block = (4, 4, 2, 2), 4, (2, 2, 1, 1)
    lat = hd.Lattice(L, Ls)
    vec = dev(planes(synth.gaussian_fermion(L, Ls, 6100, count=6)))
    sub = hd.subspace_from_vectors(lat, block, vec)
    phi = host(sub.vectors())
    pb = blocks(phi, L, Ls, block)
    v = host(dev(planes(synth.gaussian_fermion(L, Ls, 6101, count=1)))).copy()
    v[0, 5, 3, 1] = value
    with np.errstate(all="ignore"):
        want = (np.conj(pb) * blocks(v, L, Ls, block)[0]).sum(-1).T
    got = host(hd.restrict(sub, dev(v)))[0]
    fin = np.isfinite(want.real) & np.isfinite(want.imag)
    gfin = np.isfinite(got.real) & np.isfinite(got.imag)
    assert np.array_equal(fin, gfin)
    scale = np.abs(want[fin]).max()
    assert np.abs(got[fin] - want[fin]).max() <= 1e-14 * scale
    c = host(hd.restrict(sub, dev(planes(synth.gaussian_fermion(L, Ls, 6102, count=1))))).copy()
    c[0, 1, 2] = value
    with np.errstate(all="ignore"):
        wf = (pb * c[0].T[:, :, None]).sum(0)
    gf = blocks(host(hd.prolong(sub, dev(c))), L, Ls, block)[0]
    fin = np.isfinite(wf.real) & np.isfinite(wf.imag)
    assert np.array_equal(fin, np.isfinite(gf.real) & np.isfinite(gf.imag))
    if fin.any():
        other = np.delete(np.arange(wf.shape[0]), 1)
        assert np.abs(gf[other] - wf[other]).max() <= 1e-14 * np.abs(wf[other]).max()


# vector counts whose tiles fill one to six sets of threads (in fixed point up to 44) and two and three rounds
# of them, Ls for which the last chunk of 96 elements ends inside a group of 16, shares of a block
@pytest.mark.parametrize("L,Ls,block,nvec", [((4, 4, 2, 2), 3, (2, 2, 1, 1), 2), ((4, 4, 4, 4), 5, (2, 2, 2, 2), 8),
                                             ((4, 4, 4, 4), 8, (2, 2, 2, 2), 24), ((6, 2, 2, 6), 7, (3, 1, 1, 3), 34),
                                             ((4, 4, 4, 4), 3, (2, 2, 2, 2), 44), ((4, 4, 4, 4), 4, (2, 2, 2, 2), 46),
                                             ((4, 4, 4, 4), 5, (2, 2, 2, 2), 64)])
@pytest.mark.parametrize("scale", [None, "spread", "outside"])
def test_block_orthonormalisation(hd, L, Ls, block, nvec, scale):
    v = synth.gaussian_fermion(L, Ls, 6100, count=nvec)
    if scale == "spread":       # the fifth dimension's profile, and vectors of different sizes
        v = v * np.exp(-3.0 * np.arange(Ls))[:, None, None]
        v = v * 10.0 ** (np.arange(nvec) % 7 - 3.0).reshape((-1,) + (1,) * 7)
    elif scale == "outside":    # groups of one vector below the format's smallest exponent
        v[0][..., :2, :] *= 1e-220
    got = host(hd.subspace_from_vectors(hd.Lattice(L, Ls), block, dev(planes(v)), store_dtype=torch.complex128).vectors())
    q = blocks(got, L, Ls, block).astype(np.clongdouble)
    x = blocks(host(dev(planes(v))), L, Ls, block).astype(np.clongdouble)
    for a in range(q.shape[1]):
        # the second round's Gram matrix is the identity to cond(V)^2 u; its factor's inverse and the
        # product with it add nvec terms each
        gram = np.conj(q[:, a]) @ q[:, a].T
        assert np.abs(gram - np.eye(nvec)).max() <= 1.2e-16 * (16 + 2 * nvec)
        r = np.conj(q[:, a]) @ x[:, a].T
        assert (np.abs(np.tril(r, -1)).max(0) / np.sqrt((np.abs(x[:, a]) ** 2).sum(-1))).max() <= 1e-13


GRADES = {"colour": (np.array([1.0, 1e-5, 1e-10]), np.array([1e-10, 1e-5, 1.0])),
          "colour_near": (np.array([1.0, 0.1, 0.01]), np.array([0.01, 0.1, 1.0])),
          "spin": (np.array([1.0, 1.0, 1e-7, 1e-7])[:, None], np.array([1e-7, 1e-7, 1.0, 1.0])[:, None])}


@pytest.mark.parametrize("L,Ls,block,nvec", [((4, 4, 2, 4), 6, (2, 2, 1, 2), 2), ((8, 4, 4, 4), 16, (4, 2, 2, 2), 12),
                                             ((4, 4, 4, 4), 3, (2, 2, 2, 2), 18)])
@pytest.mark.parametrize("grade", ["colour", "colour_near", "spin", "imaginary", "one_site"])
def test_components_of_different_size(hd, L, Ls, block, nvec, grade):
    """Fields that are large where the basis is small: each real of the coefficients and of the
    prolonged field is as accurate as FP64 sums of its own terms."""
    vec = synth.gaussian_fermion(L, Ls, 6200, count=nvec)
    v = synth.gaussian_fermion(L, Ls, 6201, count=2)
    if grade in GRADES:
        vec, v = vec * GRADES[grade][0], v * GRADES[grade][1]
    elif grade == "imaginary":
        vec, v = vec.real + 1e-9j * vec.imag, v.real + 1e-9j * v.imag
    else:  # one 4d site of each block far larger in the field, and far smaller in the basis
        s = np.ones(tuple(L[::-1]) + (1, 1, 1))
        s[tuple(slice(None, None, b) for b in block[::-1])] = 1e9
        vec, v = vec / s, v * s
    lat = hd.Lattice(L, Ls)
    sub = hd.subspace_from_vectors(lat, block, dev(planes(vec)))
    vd = dev(planes(v))
    c = hd.restrict(sub, vd)
    f = hd.prolong(sub, c)
    phi = blocks(host(sub.vectors()), L, Ls, block).astype(np.clongdouble)
    vb = blocks(host(vd), L, Ls, block).astype(np.clongdouble)
    got = host(c).astype(np.clongdouble)

    def terms(a, b, conj):
        """exact a b (a conjugated or not) and the sum of the magnitudes of each real's terms, over the last axis."""
        s = 1 if conj else -1
        re, im = a.real * b.real + s * a.imag * b.imag, a.real * b.imag - s * a.imag * b.real
        tr, ti = np.abs(a.real * b.real) + np.abs(a.imag * b.imag), np.abs(a.real * b.imag) + np.abs(a.imag * b.real)
        return re.sum(-1), im.sum(-1), tr.sum(-1), ti.sum(-1)

    # FP64 multiply-adds: at most 2 nvec = 36 roundings (prolongation) or the few dozen of a thread (restriction) of
    # partial sums below the sum of magnitudes, 2^-53 sqrt(36) with a factor of 1.5 over the largest of many
    bound = 1e-15
    for r in range(2):
        re, im, tr, ti = terms(phi, vb[r][None], True)  # (nvec, Vc)
        assert (np.abs(got[r].real.T - re) <= bound * tr).all() and (np.abs(got[r].imag.T - im) <= bound * ti).all()
        a, b = phi.transpose(1, 2, 0), got[r][:, None, :]
        re, im, tr, ti = terms(a, b, False)
        fb = blocks(host(f), L, Ls, block)[r].astype(np.clongdouble)
        assert (np.abs(fb.real - re) <= bound * tr).all() and (np.abs(fb.imag - im) <= bound * ti).all()


@pytest.mark.parametrize("nvec", [2, 6])
def test_block_orthonormalisation_of_vectors_at_opposite_walls(hd, nvec):
    """Half of the vectors decay from one wall and half from the other, by e^-2 a site: where an orthonormal
    vector is smallest (1e-13) it comes from Gram entries of 1e-12, which must be as accurate as their own
    terms allow."""
    L, Ls, block = (4, 4, 2, 4), 16, (2, 2, 1, 2)
    s = np.arange(Ls)
    v = synth.gaussian_fermion(L, Ls, 6300, count=nvec)
    for k in range(nvec):
        v[k] *= np.exp(-2.0 * (s if k < nvec // 2 else s[::-1]))[:, None, None]
    got = blocks(host(hd.subspace_from_vectors(hd.Lattice(L, Ls), block, dev(planes(v))).vectors()), L, Ls, block)
    q = blocks(host(dev(planes(v))), L, Ls, block).astype(np.clongdouble)
    for k in range(nvec):  # modified Gram-Schmidt, twice, in extended precision
        for _ in range(2):
            for j in range(k):
                q[k] -= q[j] * (np.conj(q[j]) * q[k]).sum(-1, keepdims=True)
        q[k] /= np.sqrt((np.abs(q[k]) ** 2).sum(-1, keepdims=True))
    shape = (nvec, q.shape[1], -1, 12, Ls)
    e = np.sqrt((np.abs((got - q).reshape(shape)) ** 2).sum((1, 2, 3)))
    w = np.sqrt((np.abs(q.reshape(shape)) ** 2).sum((1, 2, 3)))
    assert (e <= 1e-13 * w).all(), e / w


def test_copy_of_the_basis_is_given_back(hd):
    """With the device's memory nearly taken, a solve's workspace that does not fit beside the fixed-point
    copies of two bases is allocated all the same, and what used a copy runs on without it."""
    L, Ls, block, M5, mf = (16, 16, 8, 8), 8, (4, 4, 4, 4), 1.8, 0.3
    lat = hd.Lattice(L, Ls)
    U = dev(synth.gauge_field((4, 4, 4, 4), 0.3, 6500).reshape(4, -1, 3, 3))
    U = U.repeat(1, lat.V4 // 256, 1, 1).contiguous()
    gen = torch.Generator(device="cuda").manual_seed(6501)
    noise = torch.randn(8, lat.V4, 12, Ls, generator=gen, device="cuda", dtype=torch.complex128)
    b = noise[0].clone()
    sub = hd.build_subspace(lat, U, noise[:4].contiguous(), M5, mf, block, order=60, lam_cut=0.5)
    other = hd.subspace_from_vectors(lat, block, noise)
    captured = hd.subspace_from_vectors(lat, block, noise)
    del noise
    co, again = hd.build_coarse_op(sub, U, M5, mf), hd.build_coarse_op(sub, U, M5, mf)
    hd.coarse_invert(co)
    hd.coarse_invert(again)
    kw = dict(tol=1e-6, max_outer=300, inner_dtype=torch.complex128)
    x0, _ = hd.hdcr_solve(co, U, b, restart=8, **kw)
    c0 = hd.restrict(other, b)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):  # keeps its copy
        out = hd.restrict(captured, b)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    field = 12 * lat.V5 * 16
    # the workspace of restart 24 takes 55 fields in one piece and 11 more, a copy 8: all but 53 are taken
    hold = torch.empty(torch.cuda.mem_get_info()[0] - 53 * field, dtype=torch.uint8, device="cuda")
    x, st = hd.hdcr_solve(again, U, b, restart=24, **kw)
    assert st["true_resid"] <= 1e-6
    assert float((x - x0).norm() / x0.norm()) <= 1e-4
    c = hd.restrict(other, b)
    assert float((c - c0).norm() / c0.norm()) <= 1e-14
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, c0)
    del hold


@pytest.mark.parametrize("Ls", [3, 4, 5])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_fp32_transfer_of_unaligned_fields(hd, Ls, nrhs):
    """A field 8 bytes off a 16-byte boundary is read one element a load: the same sums as the aligned copy's, which is
    read in pairs of elements for odd Ls as for even, to their order."""
    L, block = (4, 4, 4, 2), (2, 2, 2, 1)
    lat = hd.Lattice(L, Ls)
    sub = hd.subspace_from_vectors(lat, block, dev(planes(synth.gaussian_fermion(L, Ls, 6600, count=10))),
                                   store_dtype=torch.complex64)
    v = dev(planes(synth.gaussian_fermion(L, Ls, 6601, count=nrhs))).to(torch.complex64)
    off = torch.empty(v.numel() + 1, dtype=torch.complex64, device="cuda")[1:].view(v.shape)
    off.copy_(v)
    assert v.data_ptr() % 16 == 0 and off.data_ptr() % 16 == 8
    a, b = hd.restrict(sub, v), hd.restrict(sub, off)
    phi = blocks(host(sub.vectors()), L, Ls, block)
    want = np.stack([(np.conj(phi) * x).sum(-1).T for x in blocks(host(v), L, Ls, block)])
    for c in (a, b):  # as in test_transfer_error
        assert np.linalg.norm(host(c) - want) <= 2e-6 * np.linalg.norm(want)
    f = blocks(host(hd.prolong(sub, a)), L, Ls, block)
    wf = np.stack([(phi * x.T[:, :, None]).sum(0) for x in host(a)])
    assert np.linalg.norm(f - wf) <= 2e-6 * np.linalg.norm(wf)


@pytest.mark.parametrize("value", [1e250, 1e-250, -3e-310])
def test_results_beside_values_outside_the_format(hd, value):
    """The blocks and elements that a value outside the format reaches, each on its own scale: what is
    computed in FP64 there is the same sum, of the same terms."""
    L, Ls, block = (4, 4, 2, 2), 4, (2, 2, 1, 1)
    lat = hd.Lattice(L, Ls)
    sub = hd.subspace_from_vectors(lat, block, dev(planes(synth.gaussian_fermion(L, Ls, 6400, count=6))))
    phi = blocks(host(sub.vectors()), L, Ls, block).astype(np.clongdouble)  # (nvec, Vc, K)
    v = host(dev(planes(synth.gaussian_fermion(L, Ls, 6401, count=1)))).copy()
    v[0, 5, 3, 1] = value * (0.6 - 0.8j)
    vb = blocks(v, L, Ls, block)[0].astype(np.clongdouble)
    got = host(hd.restrict(sub, dev(v)))[0].T
    want, terms = (np.conj(phi) * vb).sum(-1), (np.abs(phi) * np.abs(vb)).sum(-1)
    # a block has 192 terms; each block and vector against its own (in extended precision, whose exponents hold them)
    assert (np.abs(got - want) <= 1e-15 * terms).all()
    c = host(hd.restrict(sub, dev(planes(synth.gaussian_fermion(L, Ls, 6402, count=1))))).copy()
    c[0, 1, 2] = value * (0.6 - 0.8j)
    got = blocks(host(hd.prolong(sub, dev(c))), L, Ls, block)[0]
    cc = c[0].T[:, :, None].astype(np.clongdouble)
    want, terms = (phi * cc).sum(0), (np.abs(phi) * np.abs(cc)).sum(0)
    assert (np.abs(got - want) <= 1e-15 * terms).all()
    # a basis vector with such a part, orthonormalised by itself
    w = synth.gaussian_fermion(L, Ls, 6403, count=2)
    w[..., 2, :, :] *= 1e-240
    sub = hd.subspace_from_vectors(lat, block, dev(planes(w)))
    phi = blocks(host(sub.vectors()), L, Ls, block).astype(np.clongdouble)
    assert (np.abs(phi[:, :, 2]) < 1e-200).all()
    vb = blocks(host(dev(planes(synth.gaussian_fermion(L, Ls, 6404, count=1)))), L, Ls, block)[0]
    vb[:, np.arange(192) % Ls != 2] = 0  # a field that meets that part alone
    n = np.zeros((1,) + vb.shape, dtype=np.complex128)
    n[0] = vb
    B, T = tuple(block[::-1]), tuple(L[::-1])
    g = [t // b for t, b in zip(T, B)]
    full = n.reshape(1, *g, *B, 12 * Ls).transpose(0, 1, 5, 2, 6, 3, 7, 4, 8, 9).reshape(1, lat.V4, 12, Ls)
    got = host(hd.restrict(sub, dev(full)))[0].T
    want, terms = (np.conj(phi) * vb).sum(-1), (np.abs(phi) * np.abs(vb)).sum(-1)
    assert (np.abs(got - want) <= 1e-15 * terms + 1e-300).all()

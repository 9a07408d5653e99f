"""Restriction over clusters of CTAs and several fields a pass, and the prolongation: error
against extended precision over block shapes, vector
counts, numbers of fields, odd and even Ls and field profiles."""
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

    # sums of up to 400 products a thread, u sqrt(n) each with u = 1.1e-16 (6e-8), over terms that
    # partly cancel
    bound = 4e-15 if dtype == "c128" else 2e-6
    assert rel(got, want) <= bound
    wf = np.stack([(phi * x.T[:, :, None]).sum(0) for x in got])
    assert rel(blocks(host(f), L, Ls, block), wf) <= bound

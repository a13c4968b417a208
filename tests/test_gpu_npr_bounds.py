"""The NPR contraction against the oracle, each hypercube within its own bound.

Scale of hypercube z: S(z) = the sum over its 256 terms of the products of absolute values (complex magnitudes of
links and fields, path averages of the links' magnitudes).  With u = 2^-53, a sum of K complex products errs by at
most 2 sqrt(2) K u of the sum of magnitudes: the path averages by 19 u, 46 u and 85 u (levels 2, 3, 4), a bilinear by
102 u, a term by 208 u and the sum of 256 by 20 u (pairwise, the GPU) or 360 u (in turn, the oracle): together below
9.2e-14 S(z).  The fixed-point form keeps the GPU's part of it.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1511_00088_gb300 import stag, synth

pytestmark = pytest.mark.gpu

BOUND = 1e-13


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1511_00088_gb300 import build
    build.build()
    stag.load()


def corner_sites(L):
    """(16, hypercubes) lexicographic sites of the corners of every hypercube."""
    H = [n // 2 for n in L]
    z = np.arange(H[0] * H[1] * H[2] * H[3])
    zc = [z % H[0], z // H[0] % H[1], z // (H[0] * H[1]) % H[2], z // (H[0] * H[1] * H[2])]
    x = [[2 * zc[m] + (a >> m & 1) for m in range(4)] for a in range(16)]
    return np.stack([y[0] + L[0] * (y[1] + L[1] * (y[2] + L[2] * y[3])) for y in x])


def scale(L, U, st, fs):
    sites = corner_sites(L)
    mag = np.abs(U)
    one = np.broadcast_to(np.eye(3), (sites.shape[1], 3, 3))
    W = {(a, a): one for a in range(16)}
    for level in range(1, 5):
        for a in range(16):
            for d in range(16):
                if bin(a ^ d).count("1") == level:
                    acc = 0
                    for m in range(4):
                        if (a ^ d) >> m & 1:
                            q = d ^ (1 << m)
                            link = mag[m][sites[min(q, d)]]
                            acc = acc + W[a, q] @ (link if d > q else np.swapaxes(link, 1, 2))
                    W[a, d] = acc / level
    f = [np.abs(v)[sites] for v in fs]  # (16, hypercubes, 3)
    S1, F1, S2, F2 = st
    out = 0
    for a in range(16):
        b = a ^ S1 ^ F1
        for c in range(16):
            d = c ^ S2 ^ F2
            out = out + (np.einsum("hi,hij,hj->h", f[0][a], W[a, d], f[3][d])
                         * np.einsum("hi,hij,hj->h", f[2][c], W[c, b], f[1][b]))
    return out


def contract(L, U, st, fs):
    with stag.Context(L) as ctx:
        ctx.links_upload(U)
        O, _ = ctx.npr_contract(st, *fs)
    return O


def check(L, U, st, fs):
    O = contract(L, U, st, fs)
    assert np.all(np.abs(O - oracle.npr_contract(L, U, *st, *fs)) <= BOUND * scale(L, U, st, fs))
    return O


@pytest.mark.parametrize("st", [(0, 0, 0, 0), (1, 2, 4, 7), (15, 15, 9, 6)])
@pytest.mark.parametrize("phases", [False, True])
def test_rows_and_columns_of_unit_norm_are_not_unitarity(st, phases):
    """Every link of rank 1 with all elements of magnitude 3^-1/2: path averages reach 3."""
    L = (4, 4, 4, 8)
    V = synth.volume(L)
    rng = np.random.default_rng(1101)
    U = np.full((4, V, 3, 3), 3 ** -0.5, np.complex128)
    if phases:  # u = a b^dag with a common b: products of forward links stay coherent
        b = np.exp(2j * np.pi * rng.uniform(size=3))
        U *= b[:, None] * np.conj(b)[None, :]
    fs = [rng.uniform(1.8, 1.99, (V, 3)) + 0j for _ in range(4)]
    check(L, U, st, fs)

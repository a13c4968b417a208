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


def spread_fields(how, V, seed):
    fs = [synth.gaussian_vector(V, seed + k) for k in range(4)]
    for k, f in enumerate(fs):
        rng = np.random.default_rng(seed + 10 + k)
        if how.startswith("corners"):
            e = int(how[7:])
            f *= 10.0 ** rng.uniform(-e, e, (V, 1))
        elif how.startswith("colours"):
            e = int(how[7:])
            f *= 10.0 ** rng.uniform(-e, e, (V, 3))
        elif how == "parts":
            f.imag *= 1e-12
    return fs


@pytest.mark.parametrize("how", ["corners4", "corners8", "corners15", "corners60", "colours8", "colours30", "parts"])
@pytest.mark.parametrize("c", [0.3, 0.4])
def test_fields_that_vary_over_a_hypercube(how, c):
    L = (4, 4, 4, 8)
    V = synth.volume(L)
    U = synth.random_links(L, c, 1111)
    for st in ((0, 0, 0, 0), (1, 2, 4, 7), (5, 10, 15, 0)):
        check(L, U, st, spread_fields(how, V, 1120))


@pytest.mark.parametrize("n", [0, 1, 2, 4])
@pytest.mark.parametrize("colours", ["plain", "apart"])
def test_single_terms(n, colours):
    """One term a hypercube: each field at one corner only, the corners of a bilinear n steps apart, its colours on
    one component each to 10^-10."""
    L = (4, 4, 4, 8)
    V = synth.volume(L)
    U = synth.random_links(L, 0.4, 1131)
    st = (0, 0, 0, 0)
    sites = corner_sites(L)
    rng = np.random.default_rng(1132)
    full = [synth.gaussian_vector(V, 1133 + k) for k in range(4)]
    fs = [np.zeros((V, 3), np.complex128) for _ in range(4)]
    for h in range(sites.shape[1]):
        A = int(rng.integers(16))
        C = A ^ int(sum(1 << m for m in rng.permutation(4)[:n]))
        for k, corner in enumerate((A, A, C, C)):  # chibar1 and chi2 at A = B, chibar3 and chi4 at C = D
            v = full[k][sites[corner, h]].copy()
            if colours == "apart":
                v *= np.where(np.arange(3) == rng.integers(3), 1.0, 1e-10)
            fs[k][sites[corner, h]] = v
    O = check(L, U, st, fs)
    assert np.all(O != 0)


@pytest.mark.parametrize("off", [0.0, 1e-9])
def test_cold_hypercubes(off):
    """Some hypercubes with (nearly) diagonal links inside a rough field, fields on one colour each to 10^-10: O(z)
    there is made of the small elements."""
    L = (4, 4, 4, 8)
    V = synth.volume(L)
    U = synth.random_links(L, 0.4, 1141)
    sites = corner_sites(L)
    rng = np.random.default_rng(1142)
    for h in (3, 17):
        for m in range(4):
            for A in range(16):
                if not A >> m & 1:
                    D = np.diag(np.exp(2j * np.pi * rng.uniform(size=3)))
                    N = rng.standard_normal((3, 3)) + 1j * rng.standard_normal((3, 3))
                    U[m, sites[A, h]] = synth.reunitarise(D + off * N)
    fs = [synth.gaussian_vector(V, 1143 + k) * np.where(np.arange(3) == k % 3, 1.0, 1e-10) for k in range(4)]
    for st in ((0, 0, 0, 0), (1, 2, 4, 7)):
        check(L, U, st, fs)


@pytest.mark.parametrize("how", ["far", "denormal", "inf", "nan", "zero_times_inf"])
def test_ends_of_the_range_on_the_integer_kernel(how):
    """Fields that leave the integer form's exponent range, on a lattice and field that it takes; a non-finite value
    stays in its hypercube."""
    L = (4, 4, 4, 8)
    V = synth.volume(L)
    U = synth.random_links(L, 0.4, 1151)
    fs = [synth.gaussian_vector(V, 1152 + k) for k in range(4)]
    st = (1, 2, 4, 7)
    if how == "far":
        fs = [f * s for f, s in zip(fs, (1e160, 1e-160, 1e140, 1e-150))]
        check(L, U, st, fs)
        return
    if how == "denormal":
        fs = [f * s for f, s in zip(fs, (1e-309, 1e290, 1e8, 1.0))]
        ref = oracle.npr_contract(L, U, *st, *fs)
        O = contract(L, U, st, fs)
        # elements of 1e-309 hold 2^-1074, 5e-15 of themselves; products of them round to that once more a term
        assert np.all(np.abs(O - ref) <= 1e-12 * scale(L, U, st, fs) + 1e-300)
        return
    clean = oracle.npr_contract(L, U, *st, *fs)
    site = int(corner_sites(L)[6, 9])
    fs[1] = fs[1].copy()
    fs[1][site, 2] = np.nan if how == "nan" else np.inf
    if how == "zero_times_inf":
        fs[0] = fs[0].copy()
        fs[0][corner_sites(L)[:, 9]] = 0.0
    O = contract(L, U, st, fs)
    bad = ~np.isfinite(O)
    assert bad.sum() == 1 and bad[9]
    S = scale(L, U, st, [np.where(np.isfinite(f), f, 0) for f in fs])
    assert np.all(np.abs(O - clean)[~bad] <= BOUND * S[~bad])


@pytest.mark.parametrize("L", [(2, 2, 2, 2), (4, 2, 6, 4), (4, 4, 4, 8)])
def test_the_forms_that_run(L, monkeypatch):
    """Rough SU(3) fields contract on the integer pipe (other bits than the FP64 form); fields that are nearly
    diagonal or not unitary in FP64 (the same bits)."""
    V = synth.volume(L)
    fs = [synth.gaussian_vector(V, 1162 + k) for k in range(4)]
    fields = {"rough": synth.random_links(L, 0.4, 1161), "cold": synth.random_links(L, 0.02, 1161),
              "unit": synth.unit_links(L), "scaled": 1.5 * synth.random_links(L, 0.4, 1161)}
    for name, U in fields.items():
        monkeypatch.delenv("STAG_FX", raising=False)
        a = contract(L, U, (1, 2, 4, 7), fs)
        monkeypatch.setenv("STAG_FX", "0")
        b = contract(L, U, (1, 2, 4, 7), fs)
        assert np.array_equal(a, b) == (name != "rough"), name

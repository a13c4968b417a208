"""The FP64 operator from fixed-point links (integer-pipe products) against the FP64 oracle.

Bound per output site: the oracle's own FP64 sums of 48 products err by at most
48 x 2^-53 of the largest neighbour component (near-unitary links), the
fixed-point sums by far less; 8e-15 of that component covers both.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1511_00088_gb300 import stag, synth

pytestmark = pytest.mark.gpu

LATTICES = [(2, 2, 2, 2), (4, 2, 6, 8), (6, 6, 6, 12), (10, 4, 2, 6)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1511_00088_gb300 import build
    build.build()
    stag.load()


def neighbour_max(L, v, par_out):
    """Largest |component| of the 8 neighbours of every site of parity par_out; v on the other parity."""
    x = np.indices(tuple(reversed(L)))[::-1].reshape(4, -1)  # x, y, z, t in lexicographic order
    par = x.sum(0) % 2
    full = np.zeros(x.shape[1])
    full[par != par_out] = np.maximum(np.abs(v.real), np.abs(v.imag)).max(1)
    grid = full.reshape(tuple(reversed(L)))
    out = np.zeros_like(grid)
    for ax in range(4):
        for d in (1, -1):
            out = np.maximum(out, np.roll(grid, d, axis=ax))
    return out.reshape(-1)[par == par_out]


def check_site_bound(L, got, ref, v, par_out):
    bound = 8e-15 * neighbour_max(L, v, par_out)[:, None]
    assert np.all(np.abs(got - ref) <= bound)


@pytest.mark.parametrize("L", LATTICES)
@pytest.mark.parametrize("spread", ["plain", "wide", "point"])
def test_half_operators_site_by_site(L, spread):
    V = synth.volume(L)
    U = synth.random_links(L, 0.4, 701)
    vs = []
    for seed in (702, 703):
        v = synth.gaussian_vector(V // 2, seed)
        rng = np.random.default_rng(seed)
        if spread == "wide":  # neighbouring sites (and components) up to 10^80 apart
            v = v * 10.0 ** rng.uniform(-40, 40, (V // 2, 1)) * 10.0 ** rng.uniform(-10, 10, (V // 2, 3))
        elif spread == "point":  # most neighbourhoods are exactly zero
            keep = np.zeros(V // 2)
            keep[rng.integers(V // 2)] = 1.0
            v = v * keep[:, None]
        vs.append(v)
    with stag.Context(L) as ctx:
        ctx.links_upload(U)
        oe = ctx.dslash_oe(torch.from_numpy(vs[0]).cuda()).cpu().numpy()
        eo = ctx.dslash_eo(torch.from_numpy(vs[1]).cuda()).cpu().numpy()
    check_site_bound(L, oe, oracle.dslash_oe(L, U, vs[0]), vs[0], 1)
    check_site_bound(L, eo, oracle.dslash_eo(L, U, vs[1]), vs[1], 0)


@pytest.mark.parametrize("scale", [1e-305, 1e-290, 1e290, 1e305])
def test_ends_of_the_exponent_range(scale):
    L = (4, 4, 2, 6)
    U = synth.random_links(L, 0.4, 711)
    v = synth.gaussian_vector(synth.volume(L) // 2, 712)
    with stag.Context(L) as ctx:
        ctx.links_upload(U)
        got = ctx.dslash_oe(v * scale)
    check_site_bound(L, got / scale, oracle.dslash_oe(L, U, v), v, 1)


def test_non_finite_inputs_stay_visible():
    """An infinity or a NaN reaches the output sites next to it and no other."""
    L = (6, 4, 4, 6)
    V = synth.volume(L)
    U = synth.random_links(L, 0.4, 721)
    v = synth.gaussian_vector(V // 2, 722)
    clean = v.copy()
    clean[17] = clean[40] = 0.0
    near = neighbour_max(L, (v - clean), 1) > 0
    v[17, 1] = np.inf
    v[40, 0] = complex(0.0, np.nan)
    with stag.Context(L) as ctx:
        ctx.links_upload(U)
        bad, ok = ctx.dslash_oe(v), ctx.dslash_oe(clean)
    assert np.all(~np.isfinite(bad[near]).all(1)) and np.array_equal(bad[~near], ok[~near])


@pytest.mark.parametrize("how", ["small", "large", "one_row", "unit"])
def test_fields_that_are_not_unitary(how):
    """Such a field runs on FP64 FMAs; a context moves between the two forms with its field."""
    L = (4, 4, 4, 6)
    V = synth.volume(L)
    U = synth.random_links(L, 0.4, 731)
    W = {"small": 1e-3 * U, "large": 30.0 * U, "one_row": U.copy(), "unit": synth.unit_links(L)}[how]
    if how == "one_row":
        W[2, 5, 1] *= 1e-9
    v = synth.gaussian_vector(V // 2, 732)
    b = synth.gaussian_vector(V // 2, 733)
    with stag.Context(L) as ctx:
        for field in (U, W, U):
            ctx.links_upload(field)
            ref = oracle.mdagm(L, field, 0.3, v)
            got = ctx.mdagm(v, 0.3)
            assert np.linalg.norm(got - ref) <= 1e-13 * np.linalg.norm(ref)
            if how != "large":
                xs, _, _, _ = ctx.cg_solve([b] * 5, [0.3], tol=1e-10, precision=stag.STAG_FP64)
                assert all(oracle.true_residual(L, field, 0.3, b, x) <= 1e-10 for x in xs)


@pytest.mark.parametrize("case", ["far", "mixed_sites", "zero", "inf"])
def test_npr_fields_off_the_integer_range(case):
    """Hypercubes whose fields leave the integer form's exponent range contract in FP64 (1e-13 of the largest |O|,
    both sides FP64); a non-finite field value stays in its hypercube."""
    L = (4, 2, 6, 4)
    V = synth.volume(L)
    U = synth.random_links(L, 0.4, 741)
    fs = [synth.gaussian_vector(V, 742 + k) for k in range(4)]
    if case == "far":
        fs = [f * s for f, s in zip(fs, (1e160, 1e-160, 1e140, 1e-150))]
    elif case == "mixed_sites":  # neighbouring corners 10^30 apart
        fs = [f * 10.0 ** np.random.default_rng(750 + k).uniform(-15, 15, (V, 1)) for k, f in enumerate(fs)]
    elif case == "zero":
        fs[2] = np.zeros_like(fs[2])
    ref = oracle.npr_contract(L, U, 1, 2, 4, 7, *fs)
    if case == "inf":
        fs[1] = fs[1].copy()
        fs[1][5, 2] = np.inf
    with stag.Context(L) as ctx:
        ctx.links_upload(U)
        O, _ = ctx.npr_contract((1, 2, 4, 7), *fs)
    if case == "inf":
        bad = ~np.isfinite(O)
        assert bad.sum() == 1 and np.abs(O - ref)[~bad].max() <= 1e-13 * np.abs(ref).max()
    else:
        assert np.abs(O - ref).max() <= 1e-13 * np.abs(ref).max()


@pytest.mark.parametrize("alpha", [(0.9, 0.9, 0.9), (0.05, 0.6, 0.3), (0.75, 0.6, 0.0), (-0.2, 1.3, 0.3)])
def test_hyp_parameters_on_both_forms(alpha):
    """Mixes the fixed-point form holds, and those it leaves to FP64 (a weight near or below zero, or above one);
    links within 1e-13 of the oracle's."""
    L = (4, 2, 6, 8)
    U = synth.random_links(L, 0.3, 761)
    ref = oracle.hyp(L, U, alpha)
    with stag.Context(L) as ctx:
        H = ctx.hyp_smear(torch.from_numpy(U).cuda(), alpha).cpu().numpy()
    assert np.abs(H - ref).max() <= 1e-13

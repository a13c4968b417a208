"""The FP64 operator's integer-pipe form, every real component of the output within the bound of an FP64 sum.

A component is a sum of 48 products; m = the sum of their magnitudes.  The fixed-point form errs by at most
98 x 2^-53 m (its guard sends every sum with m below 2^-5 of the scale to FP64), the oracle's FP64 sum by 50 x 2^-53 m:
together below 1.7e-14 m.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1511_00088_gb300 import stag, synth

pytestmark = pytest.mark.gpu

BOUND = 1.7e-14


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1511_00088_gb300 import build
    build.build()
    stag.load()


def magnitudes(L, U, v, par_out):
    """m of the real and the imaginary part of every output component of parity par_out; v on the other parity."""
    V = synth.volume(L)
    grid = tuple(reversed(L))
    x = np.indices(grid)[::-1].reshape(4, -1)
    par = x.sum(0) % 2
    full = np.zeros((V, 3), np.complex128)
    full[par != par_out] = v
    re, im = np.zeros((V, 3)), np.zeros((V, 3))

    def add(u, w):
        ur, ui, wr, wi = np.abs(u.real), np.abs(u.imag), np.abs(w.real), np.abs(w.imag)
        with np.errstate(over="ignore"):
            re[:] += np.einsum("sij,sj->si", ur, wr) + np.einsum("sij,sj->si", ui, wi)
            im[:] += np.einsum("sij,sj->si", ur, wi) + np.einsum("sij,sj->si", ui, wr)

    lex = np.arange(V).reshape(grid)
    for mu in range(4):
        fwd = np.roll(lex, -1, axis=3 - mu).reshape(-1)
        bwd = np.roll(lex, 1, axis=3 - mu).reshape(-1)
        add(U[mu], full[fwd])
        add(np.conj(np.swapaxes(U[mu][bwd], 1, 2)), full[bwd])
    return re[par == par_out], im[par == par_out]


def check(L, U, v, got, ref, par_out):
    re, im = magnitudes(L, U, v, par_out)
    assert np.all(np.abs(got.real - ref.real) <= BOUND * re)
    assert np.all(np.abs(got.imag - ref.imag) <= BOUND * im)


def links(kind, L, seed):
    V = synth.volume(L)
    rng = np.random.default_rng(seed)
    if kind == "unit":
        return synth.unit_links(L)
    if kind == "phases":  # diagonal links
        ph = np.exp(2j * np.pi * rng.uniform(size=(4, V, 3)))
        return ph[..., None] * np.eye(3)
    U = synth.random_links(L, {"rough": 0.4, "smooth": 0.1}.get(kind, 0.4), seed)
    if kind == "scaled":
        U *= 1.01
    if kind == "some_cold":  # one link in thirty nearly diagonal, off-diagonal elements of 1e-7
        cold = rng.random((4, V)) < 1 / 30
        n = int(cold.sum())
        D = np.exp(2j * np.pi * rng.uniform(size=(n, 3)))[..., None] * np.eye(3)
        U[cold] = synth.reunitarise(D + 1e-7 * (rng.standard_normal((n, 3, 3)) + 1j * rng.standard_normal((n, 3, 3))))
    return U


def vector(spread, n, seed):
    v = synth.gaussian_vector(n, seed)
    rng = np.random.default_rng(seed + 1)
    if spread == "colours":
        v = v * 10.0 ** rng.uniform(-16, 0, (n, 3))
    elif spread == "sites":
        v = v * 10.0 ** rng.uniform(-40, 40, (n, 1))
    elif spread == "parts":
        v = v.real + 1e-13j * v.imag
    elif spread == "one_colour":
        v = v * np.array([1.0, 1e-9, 1e-17])
    elif spread == "point":
        w = np.zeros_like(v)
        w[n // 3, 1] = 1.0
        v = w
    return v


@pytest.mark.parametrize("kind", ["rough", "smooth", "some_cold", "unit", "phases"])
@pytest.mark.parametrize("spread", ["plain", "colours", "sites", "parts", "one_colour", "point"])
def test_every_component_as_in_fp64(kind, spread):
    L = (6, 4, 4, 8)
    n = synth.volume(L) // 2
    U = links(kind, L, 1201)
    a, b = vector(spread, n, 1202), vector(spread, n, 1203)
    with stag.Context(L) as ctx:
        ctx.links_upload(U)
        oe, eo = ctx.dslash_oe(a), ctx.dslash_eo(b)
    check(L, U, a, oe, oracle.dslash_oe(L, U, a), 1)
    check(L, U, b, eo, oracle.dslash_eo(L, U, b), 0)


@pytest.mark.parametrize("kind,integer", [("rough", True), ("smooth", True), ("some_cold", True), ("unit", True),
                                          ("phases", True), ("scaled", False)])
def test_the_form_that_runs(kind, integer, monkeypatch):
    """Other bits than the FP64 form's where the integer form runs, the same where it does not."""
    check_form((6, 4, 4, 8), kind, integer, monkeypatch)


@pytest.mark.parametrize("L", [(2, 2, 2, 2), (4, 4, 2, 6), (4, 2, 6, 4)])
def test_small_lattices_run_the_integer_form(L, monkeypatch):
    check_form(L, "rough", True, monkeypatch)


def check_form(L, kind, integer, monkeypatch):
    U = links(kind, L, 1211)
    v = synth.gaussian_vector(synth.volume(L) // 2, 1212)
    got = []
    for fx in (None, "0"):
        if fx is not None:
            monkeypatch.setenv("STAG_FX", fx)
        with stag.Context(L) as ctx:
            ctx.links_upload(U)
            got.append(ctx.dslash_oe(v))
    assert np.array_equal(*got) == (not integer)


def test_kernel_timing_before_any_solve():
    """The timing entry point works on finite vectors before any solve, too: the same kernels, the same time (NaNs
    would take the FP64 branch at every site, eight times as long)."""
    L = (16, 16, 16, 32)
    with stag.Context(L) as ctx:
        ctx.links_upload(synth.random_links_device(L, 0.4, 1221))
        fresh = ctx.time_dslash(stag.STAG_FP64, nlaunch=20)[0]
        b = torch.from_numpy(synth.gaussian_vector(synth.volume(L) // 2, 1222)).cuda()
        ctx.cg_solve([b], [0.1], maxiter=30, precision=stag.STAG_FP64, allow_not_converged=True)
        after = ctx.time_dslash(stag.STAG_FP64, nlaunch=20)[0]
    assert 0.6 * after <= fresh <= 1.6 * after

"""The persistent CG kernel (all iterations up to a reliable update in one cooperative launch) in each of its forms,
forced with STAG_PS = lanes per site (1, 2, 4), against the oracle: every system to a true residual of 1e-10 by the
oracle's recomputation, repeated solves bit for bit, and the paths around it (cap, zero source, breakdown, a wait
that gives up, two contexts at once)."""
import os
import threading

import numpy as np
import pytest
import torch

import oracle
from paper_1511_00088_gb300 import stag, synth

pytestmark = pytest.mark.gpu

LATTICES = [(2, 2, 2, 2), (4, 2, 6, 8), (10, 4, 2, 6), (6, 6, 6, 12), (12, 12, 12, 24)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1511_00088_gb300 import build
    build.build()
    stag.load()


@pytest.fixture
def env(monkeypatch):
    def set_(**kv):
        for k, v in kv.items():
            monkeypatch.setenv(k, str(v))
    return set_


def context(L, U, recon=False):
    ctx = stag.Context(L, recon12=recon)
    ctx.links_upload(U)
    return ctx


@pytest.mark.parametrize("L", LATTICES)
@pytest.mark.parametrize("form", [1, 2, 4])
@pytest.mark.parametrize("recon", [False, True])
def test_forms_against_oracle(L, form, recon, env):
    V = synth.volume(L)
    U = synth.random_links(L, 0.4, 901)
    bs = [synth.gaussian_vector(V // 2, 902 + r) for r in range(2)]
    bs[1][: V // 2 - 1] *= 1e-6  # one site dominates the second source
    env(STAG_PS=form)
    for masses, srcs in (([0.07], bs[:1]), ([0.05, 0.3], bs)):
        with context(L, U, recon) as ctx:
            xs, _, _, tr = ctx.cg_solve(srcs, masses, tol=1e-10, maxiter=5000)
            f = ctx.solve_form()
            assert f["kernels"] == "k_cg_persist" and f["lanes_k1"] == form
            again, _, _, _ = ctx.cg_solve(srcs, masses, tol=1e-10, maxiter=5000)
        for r, b in enumerate(srcs):
            for k, m in enumerate(masses):
                j = r * len(masses) + k
                assert oracle.true_residual(L, U, m, b, xs[j]) <= 1e-10 and tr[j] <= 1e-10
                assert np.array_equal(xs[j], again[j])


def test_graph_equals_eager_and_cap_and_zero(env):
    L = (6, 6, 6, 12)
    V = synth.volume(L)
    U = synth.random_links(L, 0.4, 911)
    b = synth.gaussian_vector(V // 2, 912)
    z = np.zeros_like(b)
    got = []
    for eager in (0, 1):
        env(STAG_EAGER=eager)
        with context(L, U) as ctx:
            xs, _, it, _ = ctx.cg_solve([z, b], [0.03, 0.2])
            ys, st, jt, tr = ctx.cg_solve([b], [0.03], maxiter=7, allow_not_converged=True)
            assert ctx.solve_form()["kernels"] == "k_cg_persist"
        assert it[0] == it[1] == 0 and not xs[0].any() and not xs[1].any()
        assert st == stag.STAG_NOT_CONVERGED and jt[0] == 7
        assert abs(oracle.true_residual(L, U, 0.03, b, ys[0]) - tr[0]) <= 1e-6 * tr[0]
        got.append(xs + ys)
    for p, q in zip(*got):
        assert np.array_equal(p, q)


def test_many_systems_share_the_gpu():
    """24 systems of 4 masses: the converged ones leave their blocks to the others."""
    L = (4, 4, 4, 8)
    V = synth.volume(L)
    U = synth.random_links(L, 0.4, 921)
    bs = [synth.gaussian_vector(V // 2, 922 + r) for r in range(6)]
    masses = [0.02, 0.05, 0.1, 0.4]
    with context(L, U) as ctx:
        xs, _, it, _ = ctx.cg_solve(bs, masses)
        assert ctx.solve_form()["kernels"] == "k_cg_persist"
    for r, b in enumerate(bs):
        for k, m in enumerate(masses):
            assert oracle.true_residual(L, U, m, b, xs[4 * r + k]) <= 1e-10
        assert it[4 * r] > it[4 * r + 3]


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_source_is_a_breakdown(bad):
    L = (4, 4, 4, 8)
    U = synth.random_links(L, 0.4, 931)
    b = synth.gaussian_vector(synth.volume(L) // 2, 932)
    good = b.copy()
    b[5, 1] = bad
    with context(L, U) as ctx:
        with pytest.raises(stag.StagError) as e:
            ctx.cg_solve([b], [0.1])
        assert e.value.status == stag.STAG_ERR_BREAKDOWN
        xs, _, _, _ = ctx.cg_solve([good], [0.1])
    assert oracle.true_residual(L, U, 0.1, good, xs[0]) <= 1e-10


@pytest.mark.parametrize("form", [1, 2, 4])
def test_a_wait_that_gives_up(form, env):
    """Blocks that stop waiting for one another: STAG_ERR_TIMEOUT, and the device stays usable."""
    L = (12, 12, 12, 24)
    U = synth.random_links(L, 0.4, 941)
    b = synth.gaussian_vector(synth.volume(L) // 2, 942)
    env(STAG_PS=form, STAG_TEST_WAIT_GIVEUP=1)
    with context(L, U) as ctx:
        with pytest.raises(stag.StagError) as e:
            ctx.cg_solve([b], [0.1])
        assert e.value.status == stag.STAG_ERR_TIMEOUT
    env(STAG_TEST_WAIT_GIVEUP=0)
    with context(L, U) as ctx:
        xs, _, _, _ = ctx.cg_solve([b], [0.1])
    assert oracle.true_residual(L, U, 0.1, b, xs[0]) <= 1e-10


def test_two_contexts_on_two_streams():
    """Two threads solve on contexts of their own, each kernel wide enough for the whole GPU: the same bits as alone."""
    L = (16, 16, 16, 32)
    V = synth.volume(L)
    U = torch.from_numpy(synth.random_links(L, 0.4, 951)).cuda()
    bs = [torch.from_numpy(synth.gaussian_vector(V // 2, 952 + k)).cuda() for k in range(2)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in bs]
    ctxs = [stag.Context(L, stream=s.cuda_stream) for s in streams]
    try:
        alone = []
        for c, b in zip(ctxs, bs):
            c.links_upload(U)
            alone.append(c.cg_solve([b], [0.05])[0][0].clone())
            assert c.solve_form()["kernels"] == "k_cg_persist"
        torch.cuda.synchronize()
        got = [None, None]

        def work(k):
            out = []
            for _ in range(5):
                out.append(ctxs[k].cg_solve([bs[k]], [0.05])[0][0])
            got[k] = out
        threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        torch.cuda.synchronize()
        for k in range(2):
            assert got[k] is not None and all(torch.equal(x, alone[k]) for x in got[k])
    finally:
        for c in ctxs:
            c.close()

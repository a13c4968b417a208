"""Calls around the persistent CG kernel that the two-kernel form answers: several contexts at once, sources near the
ends of FP32's range, streams with part of the GPU, switches at their defaults, a form asked for after an upload."""
import ctypes
import threading

import numpy as np
import pytest
import torch

import oracle
from paper_1511_00088_gb300 import stag, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1511_00088_gb300 import build
    build.build()
    stag.load()


@pytest.mark.parametrize("eager", ["1", "0"])
def test_threads_with_lattices_of_different_sizes(eager, monkeypatch):
    """Two threads whose contexts run the same kernel with different amounts of shared memory."""
    monkeypatch.setenv("STAG_EAGER", eager)
    sizes = [(8, 8, 8, 8), (4, 4, 4, 4)]
    streams = [torch.cuda.Stream() for _ in sizes]
    failures = []

    def work(k):
        try:
            L = sizes[k]
            b = synth.gaussian_vector(synth.volume(L) // 2, 1302 + k)
            U = synth.random_links(L, 0.4, 1301)
            for _ in range(6):  # a graph is built for every upload
                with stag.Context(L, stream=streams[k].cuda_stream) as ctx:
                    ctx.links_upload(U)
                    for _ in range(40):
                        x = ctx.cg_solve([b], [0.3])[0][0]
                    assert ctx.solve_form()["kernels"] == "k_cg_persist" and ctx.solve_form()["lanes_k1"] == 4
            assert oracle.true_residual(L, U, 0.3, b, x) <= 1e-10
        except Exception as e:  # noqa: BLE001 (reported by the main thread)
            failures.append((k, e))
    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures


@pytest.mark.parametrize("L,scale,tol", [((16, 16, 16, 32), 1.6e17, 1e-10), ((16, 16, 16, 32), 1e-12, 1e-10),
                                         ((16, 16, 16, 32), 1e-13, 1e-10), ((8, 8, 8, 8), 1e-12, 1e-10),
                                         ((8, 8, 8, 8), 1e-17, 1e-4)])
def test_sources_near_the_ends_of_fp32(L, scale, tol, monkeypatch):
    """FP32 sums of squares near overflow, and among the denormals: both forms solve."""
    U = synth.random_links(L, 0.4, 1311)
    b = scale * synth.gaussian_vector(synth.volume(L) // 2, 1312)
    for ps in (None, "0"):
        if ps is not None:
            monkeypatch.setenv("STAG_PS", ps)
        with stag.Context(L, recon12=True) as ctx:
            ctx.links_upload(U)
            xs, _, _, _ = ctx.cg_solve([b], [0.2], tol=tol, maxiter=2000)
            assert (ctx.solve_form()["kernels"] == "k_cg_persist") == (ps is None)
        assert oracle.true_residual(L, U, 0.2, b, xs[0]) <= 1.001 * tol


def test_the_form_of_the_last_solve_outlives_an_upload():
    """stag_solve_form and stag_solve_stats describe the last solve also after a field of the other operator form."""
    L = (4, 4, 4, 8)
    U = synth.random_links(L, 0.4, 1321)
    b = synth.gaussian_vector(synth.volume(L) // 2, 1322)
    fields = (U, 2.0 * U, U)
    with stag.Context(L) as ctx:
        for k, W in enumerate(fields):
            ctx.links_upload(W)
            if k:
                assert ctx.solve_form() == form and ctx.solve_stats() == stats
            xs, _, _, _ = ctx.cg_solve([b] * 5, [0.3], precision=stag.STAG_FP64)
            assert all(oracle.true_residual(L, W, 0.3, b, x) <= 1e-10 for x in xs)
            form, stats = ctx.solve_form(), ctx.solve_stats()


@pytest.mark.parametrize("switch", ["STAG_PDL", "STAG_FOLD", "STAG_PERSIST"])
def test_a_switch_at_its_default_changes_nothing(switch, monkeypatch):
    L = (8, 8, 8, 8)
    U = synth.random_links(L, 0.4, 1331)
    b = synth.gaussian_vector(synth.volume(L) // 2, 1332)
    got = {}
    for value in ("", "1", "0"):
        monkeypatch.setenv(switch, value)
        with stag.Context(L) as ctx:
            ctx.links_upload(U)
            ctx.cg_solve([b], [0.3])
            got[value] = ctx.solve_form()["kernels"]
    assert got == {"": "k_cg_persist", "1": "k_cg_persist", "0": "k_dslash"}


class PartOfTheGpu:
    """A stream that may use some 16 SMs of the GPU (a green context), by the driver API."""

    def __enter__(self):
        torch.cuda.init()
        torch.cuda.synchronize()
        cu = ctypes.CDLL("libcuda.so.1")

        def call(name, *args):
            assert getattr(cu, name)(*args) == 0, name
        self.call, size = call, 1024  # of a resource, more than it needs
        whole, part, rest = (ctypes.create_string_buffer(size) for _ in range(3))
        dev, n = ctypes.c_int(), ctypes.c_uint(1)
        desc, self.green, self.stream = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
        call("cuDeviceGet", ctypes.byref(dev), torch.cuda.current_device())
        call("cuDeviceGetDevResource", dev, whole, 1)  # the SMs
        call("cuDevSmResourceSplitByCount", part, ctypes.byref(n), whole, rest, 0, 16)
        call("cuDevResourceGenerateDesc", ctypes.byref(desc), part, 1)
        call("cuGreenCtxCreate", ctypes.byref(self.green), desc, dev, 1)
        call("cuGreenCtxStreamCreate", ctypes.byref(self.stream), self.green, 1, 0)
        return self.stream.value

    def __exit__(self, *_):
        torch.cuda.synchronize()
        self.call("cuStreamDestroy_v2", self.stream)
        self.call("cuGreenCtxDestroy", self.green)


@pytest.mark.parametrize("L", [(8, 8, 8, 8), (12, 12, 12, 24), (16, 16, 16, 32)])
@pytest.mark.parametrize("eager", ["1", "0"])
def test_a_stream_with_part_of_the_gpu(L, eager, monkeypatch):
    """As many blocks as the stream's SMs hold."""
    monkeypatch.setenv("STAG_EAGER", eager)
    U = synth.random_links(L, 0.4, 1351)
    b = synth.gaussian_vector(synth.volume(L) // 2, 1352)
    with PartOfTheGpu() as stream:
        for masses in ([0.3], [0.3, 0.5]):
            with stag.Context(L, stream=stream) as ctx:
                ctx.links_upload(U)
                xs = ctx.cg_solve([b], masses)[0]
                ctx.solve_form()
            for m, x in zip(masses, xs):
                assert oracle.true_residual(L, U, m, b, x) <= 1e-10


def test_a_solve_whose_blocks_gave_up_is_run_again(monkeypatch):
    """Blocks of the persistent kernel that stop waiting for one another: every solve call falls back to the two-kernel
    form, also one whose solution replaces its source."""
    monkeypatch.setenv("STAG_TEST_WAIT_GIVEUP", "2")
    L, masses = (8, 8, 8, 8), [0.2, 0.4]
    V = synth.volume(L)
    U = synth.random_links(L, 0.4, 1361)
    b, f = synth.gaussian_vector(V // 2, 1362), synth.gaussian_vector(V, 1363)
    with stag.Context(L) as ctx, stag.Context((4, 4, 4, 8)) as small:
        ctx.links_upload(U)
        W = synth.random_links((4, 4, 4, 8), 0.4, 1364)
        small.links_upload(W)
        bs = synth.gaussian_vector(256, 1365)
        for _ in range(2):
            xs = ctx.cg_solve([b], masses)[0]
            assert ctx.solve_form()["kernels"] != "k_cg_persist"
            ms = ctx.cg_solve_multishift([b], masses)[0]
            (rag, ragged), (one,) = [o for o in stag.cg_solve_ragged([(ctx, [b], masses), (small, [bs], [0.2])])[0]]
            for x in (xs, ms, (rag, ragged)):
                assert all(oracle.true_residual(L, U, m, b, y) <= 1e-10 for m, y in zip(masses, x))
            assert oracle.true_residual((4, 4, 4, 8), W, 0.2, bs, one) <= 1e-10
            full = ctx.solve_full([f], masses)[0]
            for m, y in zip(masses, full):
                r = f - 2.0 * m * y - oracle.dslash_full(L, U, y)
                assert np.linalg.norm(r) <= 1e-10 * np.linalg.norm(f)
        y = torch.from_numpy(b.copy()).cuda()
        ctx.cg_solve([y], [0.2], xs=[y])
        assert oracle.true_residual(L, U, 0.2, b, y.cpu().numpy()) <= 1e-10


@pytest.mark.parametrize("nrhs,nmass,persistent", [(4, 19, True), (7, 11, False)])
def test_many_systems_with_idle_sms(nrhs, nmass, persistent):
    """76 systems get two blocks each; 77 would leave half of the SMs idle, and keep the two-kernel form."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("counts for 152 SMs")
    L = (8, 8, 8, 8)
    U = synth.random_links(L, 0.4, 1371)
    bs = [synth.gaussian_vector(synth.volume(L) // 2, 1372 + r) for r in range(nrhs)]
    masses = [0.3 + 0.05 * k for k in range(nmass)]
    with stag.Context(L) as ctx:
        ctx.links_upload(U)
        xs, _, _, tr = ctx.cg_solve(bs, masses)
        assert (ctx.solve_form()["kernels"] == "k_cg_persist") == persistent
    assert max(tr) <= 1e-10
    for r, k in ((0, 0), (nrhs - 1, nmass - 1)):
        assert oracle.true_residual(L, U, masses[k], bs[r], xs[r * nmass + k]) <= 1e-10

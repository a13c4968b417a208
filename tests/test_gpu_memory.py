"""Device memory: what a context holds, and a solve that does not fit."""
import numpy as np
import pytest
import torch

from paper_1511_00088_gb300 import stag, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1511_00088_gb300 import build
    build.build()
    stag.load()


def test_a_solve_that_does_not_fit_can_be_repeated():
    """More systems than the device holds: out of memory each time, and smaller solves after it."""
    L = (48, 48, 48, 32)
    n = synth.volume(L) // 2
    assert 4096 * n * 48 > torch.cuda.get_device_properties(0).total_memory
    links = torch.zeros((4, 2 * n, 3, 3), dtype=torch.complex128, device="cuda")
    links += torch.eye(3, dtype=torch.complex128, device="cuda")
    b = torch.from_numpy(synth.gaussian_vector(n, 1431)).cuda()
    x = torch.empty_like(b)
    with stag.Context(L) as ctx:
        ctx.links_upload(links)
        for _ in range(2):
            with pytest.raises(stag.StagError) as e:
                ctx.cg_solve([b], list(np.linspace(1.0, 2.0, 4096)), xs=[x] * 4096)
            assert e.value.status == stag.STAG_ERR_OOM
        xs, _, _, tr = ctx.cg_solve([b], [1.0, 2.0])
        for m, y, t in zip((1.0, 2.0), xs, tr):
            r = b - ctx.mdagm(y, m)
            assert torch.linalg.norm(r) <= 1.001e-10 * torch.linalg.norm(b) and t <= 1e-10


L = (16, 16, 16, 32)
FIELD = 4 * synth.volume(L) * 144  # bytes of a gauge field
SLACK = 8 << 20                    # the driver's allocation granularity


def used():
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


@pytest.mark.parametrize("scale", [1.0, 3.0])
def test_upload_holds_two_copies(scale):
    U = scale * synth.random_links_device(L, 0.4, 1401)
    x = torch.from_numpy(synth.gaussian_vector(synth.volume(L) // 2, 1402)).cuda()
    with stag.Context((4, 4, 4, 4)) as ctx:  # modules loaded
        ctx.links_upload(synth.random_links((4, 4, 4, 4), 0.4, 1))
    before = used()
    with stag.Context(L) as ctx:
        ctx.links_upload(U)
        assert used() - before <= 2 * FIELD + SLACK
        held = used()
        g, f = ctx.force(x, grad=False, lie=True)  # needs no copy of its own
        del g
        assert used() - held <= f.numel() * 8 + 3 * x.numel() * 16 + SLACK


def test_hyp_holds_two_levels():
    U = synth.random_links_device(L, 0.4, 1411)
    out = torch.empty_like(U)
    before = used()
    with stag.Context(L) as ctx:
        ctx.hyp_smear(U, out=out)
        assert used() - before <= 6 * FIELD + SLACK

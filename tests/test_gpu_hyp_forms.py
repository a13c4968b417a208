"""Which of HYP smearing's two forms runs, and the small elements of fields that hardly mix the colours."""
import numpy as np
import pytest
import torch

import oracle
from paper_1511_00088_gb300 import stag, synth

pytestmark = pytest.mark.gpu

L = (4, 4, 4, 6)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1511_00088_gb300 import build
    build.build()
    stag.load()


def smear(U, alpha=None):
    with stag.Context(L) as ctx:
        return ctx.hyp_smear(torch.from_numpy(U).cuda(), alpha).cpu().numpy()


def field(name):
    V = synth.volume(L)
    if name == "unit":
        return synth.unit_links(L)
    if name == "rank1":
        return np.full((4, V, 3, 3), 3 ** -0.5, np.complex128)
    if name == "phases":  # diagonal to 1e-9
        rng = np.random.default_rng(1602)
        D = np.exp(0.3j * rng.standard_normal((4, V, 3)))[..., None] * np.eye(3)
        return synth.reunitarise(D + 1e-9 * (rng.standard_normal(D.shape) + 1j * rng.standard_normal(D.shape)))
    U = synth.random_links(L, {"rough": 0.4, "smooth": 0.1, "cold": 0.02}[name], 1601)
    return U


@pytest.mark.parametrize("name,integer", [("rough", True), ("smooth", True), ("cold", False), ("unit", False),
                                          ("phases", False), ("rank1", False)])
def test_the_form_that_runs(name, integer, monkeypatch):
    """Other bits than the FP64 form's where the integer form runs, the same where it does not."""
    U = field(name)
    a = smear(U)
    monkeypatch.setenv("STAG_FX", "0")
    assert np.array_equal(a, smear(U), equal_nan=True) == (not integer)
    if name != "rank1":
        assert np.abs(a - oracle.hyp(L, U)).max() <= 1e-13


def test_small_elements_keep_their_bits():
    """Links diagonal to 1e-9: the off-diagonal elements of the smeared links (sums of products of them with elements
    of order one) to 1e-12 of 1e-9, against the oracle."""
    U = field("phases")
    H, ref = smear(U), oracle.hyp(L, U)
    off = ~np.eye(3, dtype=bool)
    assert np.abs(ref[..., off]).max() < 1e-7
    assert np.abs((H - ref)[..., off]).max() <= 1e-21

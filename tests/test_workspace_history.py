"""The workspace of a handle that records its ancestry, over its history: the
reverse sweep keeps the derivatives of as many steps as its bound holds, so a
longer history never gets less room than a shorter one, and what it gets
beyond the recorded history stays within the bound."""
import pytest

from paper_1310_4624_gb300 import binding as B
from paper_1310_4624_gb300 import build as cuda_build
from paper_1310_4624_gb300 import synth
from paper_1310_4624_gb300.filter import config_from_workload

STEP = 24  # bytes of derivatives per particle and step
BOUND = 4 << 30


@pytest.fixture(scope="module")
def lib():
    cuda_build.build()
    return B.load()


def _bytes(history, record, G=64, Np=16384):
    wl = synth.small_rna(G=G, Np=Np)
    return B.pf_query_workspace([config_from_workload(wl, record_ancestors=record)], history)


def test_workspace_grows_with_the_history(lib):
    """The bound is reached at 170 steps of 2^20 particles."""
    sizes = [_bytes(h, True) for h in (1, 2, 20, 128, 169, 170, 171, 172, 200, 400)]
    assert sizes == sorted(sizes), sizes


@pytest.mark.parametrize("G,Np,history", [(64, 16384, 171), (64, 16384, 400), (64, 65536, 64), (4, 1 << 20, 200),
                                          (4, 1024, 128), (1, 1, 1)])
def test_derivatives_of_the_steps_that_fit(lib, G, Np, history):
    n = G * Np
    base = _bytes(history, False, G, Np)
    seg = 1
    while seg * seg < history:
        seg += 1
    steps = max(min(history, BOUND // (STEP * n)), seg)
    ckpts = (history + seg - 1) // seg + 1
    rest = 4 * n * history + 20 * n * (max(seg, 2) + ckpts + 2)  # parents, states by slot, checkpoints, adjoints
    small = (1 << 20) + 64 * G * (history + 8)
    assert abs(_bytes(history, True, G, Np) - base - rest - STEP * n * steps) <= small

"""The general instance of the cluster resampler (merge path over windows), on
the inputs that small groups send to the lean instance: ragged sizes, ties,
NaN, groups without weight and single dominant particles.  With codes it takes
groups beyond 32768 items, without them beyond 65536; unaligned arrays too."""
import numpy as np
import pytest

import oracle as ora

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _weights(kind, G, Np, rng):
    lw = np.round(rng.normal(size=(G, Np))).astype(np.float32)
    if kind == "special":
        lw[0, :] = -np.inf
        lw[1, rng.integers(0, Np, size=Np // 7)] = np.nan
        lw[2, :] = -50.0
        lw[2, Np // 2] = 0.0
        lw[3, :] = 1.25
    return lw


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("kind", ["ties", "special"])
@pytest.mark.parametrize("Np,codes", [(32769, True), (40001, True), (70001, True), (65537, False), (70001, False),
                                      (98304, False)])
def test_merge_path_matches_oracle(Np, codes, kind, shift):
    import __graft_entry__ as ge
    from paper_1310_4624_gb300.filter import resample
    ge.build()
    G = 4
    rng = np.random.default_rng(Np + shift)
    lw = _weights(kind, G, Np, rng)
    u = rng.integers(0, 2 ** 32, size=G, dtype=np.uint64).astype(np.uint32)
    buf = torch.empty(G * Np + 4, dtype=torch.float32, device="cuda")
    view = buf[shift:shift + G * Np]
    view.copy_(torch.from_numpy(lw.ravel()))
    out = resample(view, torch.from_numpy(u.view(np.int32)).cuda(), G, Np, want_q=codes)
    anc = (out[0] if codes else out).cpu().numpy().reshape(G, Np)
    for g in range(G):
        q = ora.quantize(lw[g])
        if codes:
            assert np.array_equal(out[1].cpu().numpy().view(np.uint64).reshape(G, Np)[g], q)
        assert np.array_equal(anc[g], ora.resample(q, int(u[g]))), (g, Np)

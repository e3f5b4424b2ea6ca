"""The resampler at the sizes where a group's cluster grows from 8 to 16 CTAs
(more than 131072 items with fewer than SMs / 8 groups), bit-exact against the
oracle on both sides of the line, aligned or not, with codes or without."""
import numpy as np
import pytest

import oracle as ora

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("codes", [False, True])
@pytest.mark.parametrize("G,Np", [(1, 131069), (1, 131072), (1, 131073), (2, 131076), (3, 150001), (19, 131076)])
def test_large_groups_match_oracle(G, Np, codes):
    import __graft_entry__ as ge
    from paper_1310_4624_gb300.filter import resample
    ge.build()
    rng = np.random.default_rng(G * 1009 + Np)
    lw = rng.uniform(-30.0, 0.0, size=(G, Np)).astype(np.float32)
    lw[0, : Np // 2] = -np.inf
    lw[G - 1, Np - 1] = 9.0
    u = rng.integers(0, 2 ** 32, size=G, dtype=np.uint64).astype(np.uint32)
    out = resample(torch.from_numpy(lw.ravel()).cuda(), torch.from_numpy(u.view(np.int32)).cuda(), G, Np, want_q=codes)
    anc = (out[0] if codes else out).cpu().numpy().reshape(G, Np)
    for g in range(G):
        q = ora.quantize(lw[g])
        if codes:
            assert np.array_equal(out[1].cpu().numpy().view(np.uint64).reshape(G, Np)[g], q)
        assert np.array_equal(anc[g], ora.resample(q, int(u[g])))

"""Handles of several tracks with few large groups: those groups run on
clusters, beside the one-CTA classes of the smaller ones.  Ancestors are
compared with the oracle bit for bit, and the resampling of few large groups
must not cost a multiple of what the same groups cost in a one-track handle."""
import numpy as np
import pytest

import oracle as ora
from paper_1310_4624_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def dev():
    import __graft_entry__ as ge
    ge.build()
    return torch.device("cuda:0")


def _filter(dev, sizes, T, ess=()):
    from paper_1310_4624_gb300.filter import ParticleFilter, config_from_workload
    wls = [synth.small_rna(G=g, Np=n, H=64, W=64, T=T, seed=3, data_seed=n, mode=synth.ARNA,
                           resample_rule=1 if t in ess else 0, ess_fraction=0.7) for t, (g, n) in enumerate(sizes)]
    seqs = [synth.make_sequence(wl) for wl in wls]
    pf = ParticleFilter([config_from_workload(wl, s[1][0], track_id=t) for t, (wl, s) in enumerate(zip(wls, seqs))],
                        history=max(2, T), device=dev)
    frames = [torch.from_numpy(s[0]).to(dev) for s in seqs]
    return pf, wls, frames


@pytest.mark.parametrize("sizes", [
    ((2, 40001), (3, 2049), (3, 100), (2, 2048)),  # clusters beside all three classes
    ((1, 70000), (4, 1024), (2, 31)),              # a chunk that takes the general instance under Alg. 1's test
    ((2, 33000), (2, 65533)),                      # clusters alone
    ((1, 2049), (1, 2046)),                        # either side of one sub-chunk, off the 16-byte grid
])
@pytest.mark.parametrize("ess", [(), (0,)])
def test_ancestors_match_oracle(dev, sizes, ess):
    pf, wls, frames = _filter(dev, sizes, 3, ess)
    for k in range(3):
        pf.step([f[k] for f in frames])
        for t, wl in enumerate(wls):
            p = pf.particles(track=t)
            lw = p["logw"].cpu().numpy().reshape(wl.G, wl.Np)
            anc = p["anc"].cpu().numpy().reshape(wl.G, wl.Np)
            for g in range(wl.G):
                q = ora.quantize(lw[g])
                want = ora.resample(q, ora.resample_uniform(ora.cfg_from_workload(wl, track=t), g, k))
                if wl.resample_rule == 1 and not ora.ess_test(q, wl.ess_fraction):
                    want = np.arange(wl.Np)
                assert np.array_equal(anc[g], want + g * wl.Np), (k, t, g, wl.Np)
    pf.close()


def _resample_ms(pf, frames, T):
    best = 1e9
    for _ in range(3):
        pf.reset()
        pf.profile(True)
        for k in range(T):
            pf.step([f[k] for f in frames])
        n, ms = pf.profile_read()["resample"]
        pf.profile(False)
        best = min(best, ms / n)
    return best


@pytest.mark.parametrize("sizes,one", [(((4, 65536),) * 2, (8, 65536)), (((1, 1 << 19),) * 2, (2, 1 << 19)),
                                       (((1, 1 << 19),) + ((4, 1024),) * 20, (1, 1 << 19))])
def test_few_large_groups_cost_what_one_track_costs(dev, sizes, one):
    """Three times the one-track time leaves room for its wider clusters and
    its overlapped global step; one CTA per group took 4 to 7 times as long."""
    pf, _, frames = _filter(dev, sizes, 6)
    several = _resample_ms(pf, frames, 6)
    pf.close()
    pf, _, frames = _filter(dev, (one,), 6)
    single = _resample_ms(pf, frames, 6)
    pf.close()
    assert several <= 3.0 * single, (several, single)

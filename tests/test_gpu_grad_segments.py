"""The gradient replayed in segments, where the derivatives of all steps do not
fit the workspace's bound: tracks of a handle whose total is too large for it,
against the same tracks alone, whose derivatives are all kept."""
import numpy as np
import pytest

from paper_1310_4624_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# 2^22 particles x 24 bytes x 45 steps exceed 4 GiB; segments of 7: six and a remainder of three
T = 45


@pytest.fixture(scope="module")
def dev():
    import __graft_entry__ as ge
    ge.build()
    return torch.device("cuda:0")


def _gradient(dev, wls, seqs, track_ids):
    from paper_1310_4624_gb300.filter import ParticleFilter, config_from_workload
    pf = ParticleFilter([config_from_workload(wl, s[1][0], track_id=t, record_ancestors=True)
                         for wl, s, t in zip(wls, seqs, track_ids)], history=T, device=dev)
    fr = [torch.from_numpy(s[0]).to(dev) for s in seqs]
    steps = [[f[k] for f in fr] for k in range(T)]
    for s in steps:
        pf.step(s)
    g, z = pf.backward(steps)
    g, z = g.double().cpu().numpy(), z.cpu().numpy()
    pf.close()
    return g, z


def test_segments_equal_tracks_alone(dev):
    wls = [synth.small_rna(G=3, Np=700, H=64, W=61, mode=synth.ARNA, T=T, data_seed=1),
           synth.small_rna(G=2, Np=300, H=72, W=64, mode=synth.RNA, T=T, data_seed=2, obs_model=1),
           synth.small_rna(G=64, Np=65536, H=64, W=64, mode=synth.ARNA, T=T, data_seed=3)]
    seqs = [synth.make_sequence(wl) for wl in wls]
    g, z = _gradient(dev, wls, seqs, (0, 1, 2))
    assert np.all(np.isfinite(g))
    for t in (0, 1):
        g1, z1 = _gradient(dev, wls[t:t + 1], seqs[t:t + 1], (t,))
        # the same FP32 terms; only the order of the atomic sums differs
        assert np.all(np.abs(g[t] - g1[0]) <= 1e-5 * np.abs(g1[0]).max()), (g[t], g1[0])
        assert abs(z[t] - z1[0]) <= 1e-6 * abs(z1[0])

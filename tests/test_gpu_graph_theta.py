"""Parameters set between graph steps: the captured step of a single track
holds them in its launch arguments, so it is captured anew."""
import numpy as np
import pytest

from paper_1310_4624_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("tracks", [1, 2])
def test_graph_steps_follow_set_theta(tracks):
    import __graft_entry__ as ge
    from paper_1310_4624_gb300.filter import ParticleFilter, config_from_workload
    ge.build()
    dev = torch.device("cuda:0")
    wls = [synth.small_rna(G=3, Np=500, H=48, W=52, mode=synth.ARNA, T=4, data_seed=t) for t in range(tracks)]
    seqs = [synth.make_sequence(wl) for wl in wls]
    cfgs = [config_from_workload(wl, s[1][0], track_id=t) for t, (wl, s) in enumerate(zip(wls, seqs))]
    fr = [torch.from_numpy(s[0]).to(dev) for s in seqs]
    results = []
    for graph in (True, False):
        pf = ParticleFilter(cfgs, history=4, device=dev)
        table = pf.frame_table(fr)
        for scale in (1.0, 1.2):
            for t, wl in enumerate(wls):
                pf.set_theta([scale * wl.sigma_psf, wl.amplitude, wl.background, scale * wl.sigma_pos, wl.sigma_v], track=t)
            pf.reset()
            for k in range(4):
                if graph:
                    pf.step_table(table, graph=True)
                else:
                    pf.step([f[k] for f in fr])
        results.append([x.cpu().numpy() for t in range(tracks) for p in [pf.particles(track=t)]
                        for x in (p["states"], p["anc"], p["logw"])] + [pf.estimate()[1]])
        pf.close()
    for x, y in zip(*results):
        assert np.array_equal(x, y)

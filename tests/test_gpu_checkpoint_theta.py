"""A checkpoint of a filter whose parameters were set after its creation: the
restored filter, created with the original configuration, goes on with the
saved parameters, forward and in the gradient."""
import numpy as np
import pytest

from paper_1310_4624_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("tracks", [1, 2])
def test_restored_filter_has_the_saved_parameters(tracks):
    import __graft_entry__ as ge
    from paper_1310_4624_gb300.filter import ParticleFilter, config_from_workload
    ge.build()
    dev = torch.device("cuda:0")
    wls = [synth.small_rna(G=3, Np=500, H=48, W=52, mode=synth.ARNA, T=6, data_seed=t) for t in range(tracks)]
    seqs = [synth.make_sequence(wl) for wl in wls]
    cfgs = [config_from_workload(wl, s[1][0], track_id=t, record_ancestors=True)
            for t, (wl, s) in enumerate(zip(wls, seqs))]
    fr = [torch.from_numpy(s[0]).to(dev) for s in seqs]
    steps = [[f[k] for f in fr] for k in range(6)]

    def go_on(pf, lo):
        for s in steps[lo:]:
            pf.step(s)
        out = [x for t in range(tracks) for p in [pf.particles(track=t)] for x in (p["states"], p["anc"], p["logw"])]
        grad, z = pf.backward(steps)
        return [x.cpu().numpy() for x in out] + [pf.estimate()[1], z.cpu().numpy()], grad.double().cpu().numpy()

    a = ParticleFilter(cfgs, history=6, device=dev)
    for t, wl in enumerate(wls):
        a.set_theta([1.1 * wl.sigma_psf, 0.9 * wl.amplitude, wl.background + 0.5, 1.2 * wl.sigma_pos, 1.3 * wl.sigma_v], track=t)
    a.reset()
    for s in steps[:3]:
        a.step(s)
    ck = a.save()
    ref, gref = go_on(a, 3)
    b = ParticleFilter(cfgs, history=6, device=dev)
    b.load(ck)
    out, g = go_on(b, 3)
    for x, y in zip(out, ref):
        assert np.array_equal(x, y)
    assert np.all(np.abs(g - gref) <= 1e-5 * np.abs(gref).max(axis=1, keepdims=True))
    # and a restart of it draws from the saved parameters too
    a.reset()
    b.reset()
    for x, y in zip(go_on(b, 0)[0], go_on(a, 0)[0]):
        assert np.array_equal(x, y)
    a.close()
    b.close()

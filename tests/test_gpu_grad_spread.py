"""The gradient of a spread population (the sharing start), whose tiles do not
fit a staging box and read the frame: against the FP64 oracle on the same
ancestry, over the patch radii, both observation models, odd frames, one
track (the caller's frame) and several (padded frames); and its time against
the gradient of the same population started at a point."""
import time

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


PSF = {1: 0.6, 2: 0.8, 3: 1.0, 4: 1.2, 5: 1.5, 6: 1.8, 7: 2.1}


def _filters(dev, wls):
    from paper_1310_4624_gb300.filter import ParticleFilter, config_from_workload
    seqs = [synth.make_sequence(wl) for wl in wls]
    T = wls[0].T
    pf = ParticleFilter([config_from_workload(wl, s[1][0], track_id=t, record_ancestors=True)
                         for t, (wl, s) in enumerate(zip(wls, seqs))], history=T, device=dev)
    fr = [torch.from_numpy(s[0]).to(dev) for s in seqs]
    parents = [np.tile(np.arange(wl.N, dtype=np.int32), (T, 1)) for wl in wls]
    for k in range(T):
        pf.step([f[k] for f in fr])
        for t in range(len(wls)):
            if k > 0:
                parents[t][k] = pf.particles(track=t, parents=True)["parent"].cpu().numpy()
    return pf, seqs, fr, parents


@pytest.mark.parametrize("tracks", [1, 2])
@pytest.mark.parametrize("R,obs_model", [(1, 0), (2, 1), (3, 0), (4, 0), (5, 0), (5, 1), (6, 1), (7, 0), (7, 1)])
def test_spread_gradient_matches_fp64_oracle(dev, tracks, R, obs_model):
    """Tolerances: those of the gradient's other comparisons with this oracle
    (FP32 sums of the same terms)."""
    from parity_util import _init
    wls = [synth.sharing(G=3 + t, Np=520 - 13 * t, H=70, W=83 - t, mode=synth.ARNA, T=4, seed=2, data_seed=5 + t,
                         patch_radius=R, sigma_psf=PSF[R], obs_model=obs_model, truth_noise=True)
           for t in range(tracks)]
    pf, seqs, fr, parents = _filters(dev, wls)
    grad, lz = pf.backward([[f[k] for f in fr] for k in range(4)])
    for t, wl in enumerate(wls):
        kind, x0, lo, hi, rad = _init(wl, seqs[t][1][0])
        lz_o, g_o = ora.replay_grad(ora.cfg_from_workload(wl, track=t), kind, x0, seqs[t][0], wl.T, parents[t], lo, hi,
                                    rad)
        g = grad[t].double().cpu().numpy()
        assert abs(float(lz[t]) - lz_o) <= 1e-5 * abs(lz_o), (float(lz[t]), lz_o)
        scale = np.abs(g_o).max()
        for q in range(5):
            assert abs(g[q] - g_o[q]) <= 1e-3 * abs(g_o[q]) + 1e-5 * scale, (t, ora.THETA[q], g[q], g_o[q])
    pf.close()


def test_spread_gradient_costs_a_few_staged_ones(dev):
    """Two frames of 64 x 16384 particles: reading patches from the frame
    takes about 2.8 times the staged time (1.7 against the prepared frames of
    an earlier form); with the patch arrays in local memory it took 7."""
    def backward_ms(make):
        wl = make(G=64, Np=16384, H=512, W=512, mode=synth.ARNA, T=2, seed=3, data_seed=7)
        from paper_1310_4624_gb300.filter import ParticleFilter, config_from_workload
        frames, truth = synth.make_sequence(wl)
        pf = ParticleFilter([config_from_workload(wl, truth[0], record_ancestors=True)], history=2, device=dev)
        fr = torch.from_numpy(frames).to(dev)
        for k in range(2):
            pf.step(fr[k])
        best = 1e9
        for _ in range(4):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            pf.backward([fr[0], fr[1]])
            best = min(best, time.perf_counter() - t0)
        pf.close()
        return best * 1e3

    spread, point = backward_ms(synth.sharing), backward_ms(synth.small_rna)
    assert spread <= 4.5 * point, (spread, point)

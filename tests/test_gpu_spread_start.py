"""A population that starts spread: for its first steps, method variants and
frames that no TMA descriptor can describe take the prepared frame (whose
patches need no bounds checks), then the caller's.  Which steps prepare is read
off the launch counts; the results are the same bits either way (the frame
table's route always prepares)."""
import numpy as np
import pytest

from paper_1310_4624_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

T = 11


@pytest.fixture(scope="module")
def dev():
    import __graft_entry__ as ge
    ge.build()
    return torch.device("cuda:0")


def _run(dev, wl, table):
    from paper_1310_4624_gb300.filter import ParticleFilter, config_from_workload
    frames, truth = synth.make_sequence(wl)
    fr = torch.from_numpy(frames).to(dev)
    pf = ParticleFilter([config_from_workload(wl, truth[0])], history=T, device=dev)
    tab = pf.frame_table([fr])
    pf.profile(True)
    out = []
    for k in range(T):
        if table:
            pf.step_table(tab)
        else:
            pf.step(fr[k])
        p = pf.particles()
        x, z, _ = pf.estimate()
        out += [p["states"].cpu().numpy(), p["anc"].cpu().numpy(), p["logw"].cpu().numpy(), x, z]
    prepared = pf.profile_read()["frame_prep"][0]
    pf.close()
    return out, prepared


CASES = [("ess", dict(H=96, W=128, resample_rule=1), 8),
         ("keyed", dict(H=96, W=128, send_rule=1, ex_ratio=0.3), 8),
         ("odd", dict(H=97, W=101), 8),
         ("odd_r7", dict(H=97, W=101, patch_radius=7, sigma_psf=2.1), 8),
         ("ess_r6", dict(H=97, W=101, patch_radius=6, sigma_psf=1.8, resample_rule=1), 8),
         ("tma", dict(H=96, W=128), 0),
         ("tma_r7", dict(H=96, W=128, patch_radius=7, sigma_psf=2.1), 0)]


@pytest.mark.parametrize("start", ["sharing", "point", "uniform"])
@pytest.mark.parametrize("name,kw,steps", CASES, ids=[c[0] for c in CASES])
def test_route_and_results_of_a_start(dev, name, kw, steps, start):
    wl = synth.sharing(G=3, Np=700, mode=synth.ARNA, T=T, seed=4, **kw)
    if start == "point":
        wl = wl.replace(init=synth.INIT_POINT)
    elif start == "uniform":  # never gathers within these steps: the caller's frame, off the box
        wl = wl.replace(init=synth.INIT_UNIFORM)
    a, prepared = _run(dev, wl, False)
    assert prepared == (0 if start == "point" else steps)
    b, prepared = _run(dev, wl, True)
    assert prepared == T
    for x, y in zip(a, b):
        assert np.array_equal(x, y, equal_nan=True)


def test_a_restart_is_a_start(dev):
    from paper_1310_4624_gb300.filter import ParticleFilter, config_from_workload
    wl = synth.sharing(G=3, Np=300, H=97, W=101, mode=synth.ARNA, T=T)
    frames, truth = synth.make_sequence(wl)
    fr = torch.from_numpy(frames).to(dev)
    pf = ParticleFilter([config_from_workload(wl, truth[0])], history=T, device=dev)
    for _ in range(2):
        pf.profile(True)
        for k in range(T):
            pf.step(fr[k])
        assert pf.profile_read()["frame_prep"][0] == 8
        pf.reset()
    pf.close()

"""The two launches of a one-track step overlap (the resampler starts beside
the propagate kernel's last tiles, and the next step's beside the resampler's)
also where the groups are so large that the general resampler instance runs:
a step takes less than its two kernels timed apart."""
import time

import numpy as np
import pytest

from paper_1310_4624_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("rule,G,Np", [(1, 3, 65537), (1, 2, 131072), (0, 2, 131072), (0, 16, 16384)])
def test_launches_of_a_step_overlap(rule, G, Np):
    import __graft_entry__ as ge
    from paper_1310_4624_gb300.filter import ParticleFilter, config_from_workload
    ge.build()
    T = 20
    wl = synth.small_rna(G=G, Np=Np, H=256, W=256, T=T, mode=synth.ARNA, resample_rule=rule)
    frames, truth = synth.make_sequence(wl)
    fr = torch.from_numpy(frames).cuda()
    pf = ParticleFilter([config_from_workload(wl, truth[0])], history=T)
    step = 1e9
    for _ in range(5):
        pf.reset()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for k in range(T):
            pf.step(fr[k])
        torch.cuda.synchronize()
        step = min(step, (time.perf_counter() - t0) / T * 1e3)
    apart = 1e9
    for _ in range(3):
        pf.profile(True)
        pf.reset()
        for k in range(T):
            pf.step(fr[k])
        r = pf.profile_read()
        pf.profile(False)
        apart = min(apart, sum(r[k][1] / r[k][0] for k in ("propagate_weight", "resample")))
    assert np.isfinite(pf.estimate()[1]).all()
    pf.close()
    assert step <= apart, (step, apart)

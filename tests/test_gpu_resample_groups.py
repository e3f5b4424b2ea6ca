"""The one-CTA (one-warp) per group resampler of batches against the oracle,
at the edges of its classes of group size (256, 1024 and 2048 items, with the
3 elements of padding of groups off the 16-byte grid), and the lean cluster
resampler at its largest chunk and on unaligned arrays: codes are exact
integers, so ancestors are compared bit for bit."""
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


@pytest.mark.parametrize("sizes", [(1, 31, 253, 254, 256, 257), (1021, 1022, 1024, 1025, 5), (2045, 2046, 2048, 2049, 4099),
                                   (256, 1024, 2048, 4096, 16384)])
@pytest.mark.parametrize("spread", [False, True])
def test_batch_ancestors_match_oracle(dev, sizes, spread):
    """spread: the sharing start, whose weights concentrate on a few
    particles, so that one sub-chunk's outputs fill many windows."""
    from paper_1310_4624_gb300.filter import ParticleFilter, config_from_workload
    make = synth.sharing if spread else synth.small_rna
    wls = [make(G=3, Np=n, H=64, W=64, T=3, seed=3, data_seed=n, mode=synth.ARNA) for n in sizes]
    if not spread:
        wls[1] = wls[1].replace(resample_rule=1, ess_fraction=0.7)
    seqs = [synth.make_sequence(wl) for wl in wls]
    pf = ParticleFilter([config_from_workload(wl, s[1][0], track_id=t) for t, (wl, s) in enumerate(zip(wls, seqs))],
                        device=dev)
    for k in range(3):
        pf.step([torch.from_numpy(s[0][k]).to(dev) for s in seqs])
        for t, wl in enumerate(wls):
            p = pf.particles(track=t)
            lw = p["logw"].cpu().numpy().reshape(wl.G, wl.Np)
            anc = p["anc"].cpu().numpy().reshape(wl.G, wl.Np)
            for g in range(wl.G):
                q = ora.quantize(lw[g])
                u = ora.resample_uniform(ora.cfg_from_workload(wl, track=t), g, k)
                want = ora.resample(q, u)
                if wl.resample_rule == 1 and not ora.ess_test(q, wl.ess_fraction):
                    want = np.arange(wl.Np)
                assert np.array_equal(anc[g], want + g * wl.Np), (k, t, g, wl.Np)
    pf.close()


@pytest.mark.parametrize("G,Np", [(2, 65536), (3, 65533), (2, 40001), (5, 4093), (5, 4094), (4, 8185)])
@pytest.mark.parametrize("shift", [0, 1, 3])
def test_unaligned_and_large_lean_chunks_match_oracle(dev, G, Np, shift):
    from paper_1310_4624_gb300.filter import resample
    rng = np.random.default_rng(Np + shift)
    lw = (rng.normal(size=(G, Np)) * 3.0 - 100.0).astype(np.float32)
    lw[0, Np // 3] = 0.0  # one dominant particle
    u = rng.integers(0, 2 ** 32, size=G, dtype=np.uint64).astype(np.uint32)
    buf = torch.empty(G * Np + 4, dtype=torch.float32, device=dev)
    view = buf[shift:shift + G * Np]
    view.copy_(torch.from_numpy(lw.ravel()))
    anc = resample(view, torch.from_numpy(u.view(np.int32)).to(dev), G, Np).cpu().numpy().reshape(G, Np)
    for g in range(G):
        assert np.array_equal(anc[g], ora.resample(ora.quantize(lw[g]), int(u[g]))), (G, Np, shift, g)

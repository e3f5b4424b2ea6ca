"""Where the kernels take their pixels from: a single track's frame by TMA, by
plain loads (rows off the 16-byte grid, frames smaller than a staging box, an
unaligned pointer) or, for patches that do not fit one box, straight from the
frame; and the gradient's replay from the caller's frame (one track), from
padded frames (several) and in segments."""
import numpy as np
import pytest

from paper_1310_4624_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def dev():
    import __graft_entry__ as ge
    ge.build()
    return torch.device("cuda:0")


def _device_frames(dev, frames, shift):
    """(T, H, W) on the device, each frame `shift` floats off a 16-byte boundary."""
    T, H, W = frames.shape
    out = []
    for k in range(T):
        flat = torch.zeros(H * W + 4, dtype=torch.float32, device=dev)
        flat[shift:shift + H * W] = torch.from_numpy(frames[k]).to(dev).reshape(-1)
        out.append(flat[shift:shift + H * W].view(H, W))
    return out


CASES = [("odd_rows", synth.small_rna(G=3, Np=300, H=41, W=53), 0),
         ("tiny_frame", synth.small_rna(G=2, Np=200, H=13, W=17, margin=2.0), 0),
         ("unaligned", synth.small_rna(G=3, Np=513, H=48, W=64), 1),
         ("wide_patch", synth.small_rna(G=2, Np=700, H=45, W=63, patch_radius=7, sigma_psf=2.1), 0),
         ("keyed_odd", synth.small_rna(G=5, Np=257, H=50, W=45, mode=synth.ARNA, ex_ratio=0.3, send_rule=1), 0),
         ("ess_odd", synth.small_rna(G=4, Np=512, H=50, W=47, mode=synth.ARNA, resample_rule=1, ess_fraction=0.5), 0),
         ("spread_vectors", synth.sharing(G=4, Np=512, H=96, W=128, mode=synth.ARNA), 0),
         ("spread_vectors_r7", synth.sharing(G=3, Np=400, H=100, W=120, mode=synth.RNA, patch_radius=7, sigma_psf=2.1), 0),
         ("spread_odd", synth.sharing(G=4, Np=512, H=97, W=101, mode=synth.ARNA), 0)]


@pytest.mark.parametrize("name,wl,shift", CASES, ids=[c[0] for c in CASES])
def test_step_matches_oracle(dev, name, wl, shift):
    from parity_util import run_and_compare
    from paper_1310_4624_gb300.filter import ParticleFilter, config_from_workload
    frames, truth = synth.make_sequence(wl, T=4)
    pf = ParticleFilter([config_from_workload(wl, truth[0], record_ancestors=True)], history=4, device=dev)
    run_and_compare(pf, wl, frames, truth[0], 4, _device_frames(dev, frames, shift))
    pf.close()


def _gradient(dev, wls, seqs, history):
    from paper_1310_4624_gb300.filter import ParticleFilter, config_from_workload
    pf = ParticleFilter([config_from_workload(wl, seqs[t][1][0], track_id=wl.data_seed, record_ancestors=True)
                         for t, wl in enumerate(wls)], history=history, device=dev)
    fr = [torch.from_numpy(s[0]).to(dev) for s in seqs]
    steps = [[f[k] for f in fr] for k in range(wls[0].T)]
    for s in steps:
        pf.step(s)
    g, z = pf.backward(steps)
    g, z = g.double().cpu().numpy(), z.cpu().numpy()
    pf.close()
    return g, z


def _agree(a, b):
    # the same FP32 terms; only the order of the atomic sums differs
    assert np.all(np.abs(a - b) <= 1e-5 * np.abs(b).max(axis=-1, keepdims=True)), (a, b)


def test_gradient_of_a_batch_equals_tracks_alone(dev):
    wls = [synth.small_rna(G=3, Np=700, H=48, W=51, mode=synth.ARNA, T=5, data_seed=1),
           synth.small_rna(G=2, Np=300, H=40, W=44, mode=synth.RNA, T=5, data_seed=2, obs_model=1)]
    seqs = [synth.make_sequence(wl) for wl in wls]
    g, z = _gradient(dev, wls, seqs, 5)
    for t in range(2):
        g1, z1 = _gradient(dev, wls[t:t + 1], seqs[t:t + 1], 5)
        _agree(g[t], g1[0])
        assert abs(z[t] - z1[0]) <= 1e-6 * abs(z1[0])


def test_gradient_in_segments_equals_one_pass(dev):
    """A history whose derivatives exceed the workspace bound (1048576
    particles x 200 steps x 24 B > 4 GiB) is replayed in segments of
    ceil(sqrt T) steps: three full ones and a remainder for T = 17."""
    wl = synth.differentiable(T=17)
    seqs = [synth.make_sequence(wl)]
    g, z = _gradient(dev, [wl], seqs, 200)
    g1, z1 = _gradient(dev, [wl], seqs, 17)
    _agree(g, g1)
    assert abs(z[0] - z1[0]) <= 1e-9 * abs(z1[0])

"""Checkpoints of several tracks in one handle: the resampler that the saved
filter used (one CTA per group, clusters, or both; the CTA size whose order
the carried weights' sum follows) comes back with it, whatever the new handle
would have chosen, so that a resumed filter continues bit for bit."""
import struct

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


def _snap(pf):
    out = []
    for t in range(pf.n_tracks):
        p = pf.particles(track=t)
        st = pf.stats(pf.steps - 1, track=t)
        out += [p["states"].cpu().numpy(), p["anc"].cpu().numpy(), p["logw"].cpu().numpy(), st["logW"],
                st["group_xhat"], st["group_ess"]]
    x, lz, _ = pf.estimate()
    return out + [x, lz]


# more groups than a small CTA has threads: the sum over them depends on the
# CTA size; groups of more tiles than a CTA has threads: so do the estimates
SIZES = {"many_groups": ((300, 64), (200, 61)), "large_groups": ((1, 140001), (2, 700))}


def _make(dev, sizes):
    from paper_1310_4624_gb300.filter import ParticleFilter, config_from_workload
    wls = [synth.sharing(G=g, Np=n, H=64, W=64, mode=synth.ARNA, T=8, seed=4, data_seed=t)
           for t, (g, n) in enumerate(sizes)]
    seqs = [synth.make_sequence(wl) for wl in wls]
    cfgs = [config_from_workload(wl, s[1][0], track_id=t) for t, (wl, s) in enumerate(zip(wls, seqs))]
    frames = [torch.from_numpy(s[0]).to(dev) for s in seqs]
    return (lambda: ParticleFilter(cfgs, history=8, device=dev)), frames


def _steps(pf, frames, lo, hi):
    out = []
    for k in range(lo, hi):
        pf.step([f[k] for f in frames])
        out.append(_snap(pf))
    return out


def _same(a, b):
    for x, y in zip(a, b):
        for u, v in zip(x, y):
            assert np.array_equal(u, v, equal_nan=True)


@pytest.mark.parametrize("sizes", sorted(SIZES))
@pytest.mark.parametrize("saver,loader", [(None, "128"), (None, "512"), ("128", None), ("512", None), (None, None)])
def test_resumed_batch_continues_bit_for_bit(dev, monkeypatch, sizes, saver, loader):
    """saver, loader: the resampler's CTA size forced in either handle (PFARNA_RS_THREADS), or its own choice."""
    make, frames = _make(dev, SIZES[sizes])

    def handle(force):
        if force:
            monkeypatch.setenv("PFARNA_RS_THREADS", force)
        else:
            monkeypatch.delenv("PFARNA_RS_THREADS", raising=False)
        return make()

    a = handle(saver)
    _steps(a, frames, 0, 3)
    ck = a.save()
    ref = _steps(a, frames, 3, 8)
    b = handle(loader)
    b.load(ck)
    _same(_steps(b, frames, 3, 8), ref)
    a.close()
    b.close()


def test_first_header_form_is_still_read(dev, monkeypatch):
    """A checkpoint whose header ends at the CTA size: the cluster kernel of
    that size goes on, as it was the only one when such files were written."""
    make, frames = _make(dev, SIZES["many_groups"])
    monkeypatch.setenv("PFARNA_RS_THREADS", "512")
    a = make()
    _steps(a, frames, 0, 3)
    ck = bytes(a.save())
    ref = _steps(a, frames, 3, 8)
    old = bytearray(struct.pack("<Q", 0x6b70635f666e7270) + ck[8:48] + ck[64:])
    monkeypatch.delenv("PFARNA_RS_THREADS")
    b = make()
    b.load(old)
    assert b.steps == 3
    _same(_steps(b, frames, 3, 8), ref)
    a.close()
    b.close()


def test_damaged_shapes_are_refused(dev):
    from paper_1310_4624_gb300 import binding as B
    make, frames = _make(dev, SIZES["large_groups"])
    a = make()
    _steps(a, frames, 0, 1)
    ck = a.save()
    for at, value in ((52, 99), (56, 9), (60, 96)):
        bad = bytearray(ck)
        bad[at:at + 4] = struct.pack("<i", value)
        with pytest.raises(B.PFError):
            a.load(bad)
    a.load(ck)
    _steps(a, frames, 1, 2)
    a.close()


@pytest.mark.parametrize("threads", [128, 512])
def test_weight_sum_does_not_depend_on_the_kernel(dev, threads):
    """The same filter continued by the one-CTA classes and by the cluster
    kernel (as the autotuner may choose it, at either CTA size): the carried
    weights' sum keeps its order."""
    make, frames = _make(dev, SIZES["many_groups"])
    a = make()
    _steps(a, frames, 0, 3)
    ck = a.save()
    ref = _steps(a, frames, 3, 8)
    tuned = bytearray(ck)
    tuned[40:52] = struct.pack("<iii", 1, threads, 0)  # cluster, CTA size, not by class
    b = make()
    b.load(tuned)
    _same(_steps(b, frames, 3, 8), ref)
    a.close()
    b.close()

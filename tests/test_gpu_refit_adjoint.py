"""The adjoint's kernels where their work is cut: tracks of one station up to
past the checkpoint segments' and the staging groups' edges, a map too large for
accumulators in shared memory, and more tracks than one chunk of step records."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2601_20569_gb300 import synth
from paper_2601_20569_gb300.options import TrackerOptions
from tests.test_gpu_refit import RX, device_tracks, host_tracks

pytestmark = pytest.mark.gpu


def tracked(n_primaries, **kw):
    import torch

    from paper_2601_20569_gb300 import tpc

    f = synth.generate("central_event", distort=True, n_primaries=n_primaries)
    opts = TrackerOptions().as_dict()
    tr = tpc.Tracker(RX, opts, mode=0, **({"cap_clusters": f.n} | kw))
    coeff = torch.as_tensor(f.map).cuda()
    tr.set_map(coeff)
    dev = tr.to_device(f.y, f.z, f.q, f.row, f.sector)
    tr.track(*dev)
    tracks = {k: tr.result()[k].clone() for k in ("cl_offset", "cl_ids", "params", "x", "sector")}
    return f, opts, tr, dev, coeff, tracks


@pytest.mark.parametrize("shape", [(20, 16, 18), (20, 24, 20)])  # the second: 230,400 bytes of FP64
def test_adjoint_track_lengths_and_map_sizes(shape):
    """Against the FP64 tape of the same frozen function; the bound is that of
    the whole event's adjoint (FP32 forward states, 1e-7 relative per step)."""
    import torch

    f, opts, tr, dev, _, tracks = tracked(600)
    rng = np.random.default_rng(11)
    dmap = (0.05 * rng.standard_normal((3,) + shape)).astype(np.float32)
    h = host_tracks(tracks)
    want = [1, 2, 15, 16, 17, 31, 32, 33, 47, 48, 49, 64, 65, 96, 97, 160]
    n = np.diff(h["offset"])
    cut = np.minimum(n, np.resize(want, len(n)))
    ids = np.concatenate([h["ids"][o:o + c] for o, c in zip(h["offset"], cut)])
    h = dict(h, ids=ids, offset=np.concatenate([[0], np.cumsum(cut)]).astype(np.int32))
    coeff = torch.as_tensor(dmap).cuda()
    w = rng.uniform(0.5, 1.5, len(cut))
    out = tr.refit(dev, device_tracks(h), coeff)
    r = oracle.refit(f.y, f.z, f.row, f.sector, RX, opts, h, dist_map=dmap, mode="f32")
    assert np.array_equal(out["n_clusters"].cpu().numpy(), r["rf_n"])
    g = tr.refit_backward(torch.as_tensor(w, dtype=torch.float32).cuda()).cpu().numpy().ravel()
    tape = oracle.refit(f.y, f.z, f.row, f.sector, RX, opts, h, dist_map=dmap, frozen=r, weights=w,
                        mode="tape")["grad"]
    assert np.linalg.norm(g - tape) < 5e-3 * np.linalg.norm(tape)


def test_adjoint_over_chunks_of_tracks():
    """The same tracks ten times over (more than one chunk): ten times the gradient.
    Each side is an FP64 sum rounded once to FP32, 2^-24 relative each."""
    import torch

    f, opts, tr, dev, coeff, tracks = tracked(1500, cap_clusters=3_500_000)
    nt, nr, rep = int(tracks["params"].shape[0]), int(tracks["cl_ids"].shape[0]), 10
    assert rep * nt > 32768
    many = {k: tracks[k].repeat((rep,) + (1,) * (tracks[k].dim() - 1))
            for k in ("cl_ids", "params", "x", "sector")}
    step = torch.arange(rep, device="cuda", dtype=torch.int32)[:, None] * nr
    many["cl_offset"] = torch.cat([(tracks["cl_offset"][:-1] + step).reshape(-1),
                                   torch.tensor([rep * nr], device="cuda", dtype=torch.int32)])
    one = tr.refit(dev, tracks, coeff)["chi2"].clone()
    g1 = tr.refit_backward(torch.ones(nt, device="cuda")).cpu().numpy().astype(np.float64)
    all_ = tr.refit(dev, many, coeff)["chi2"]
    assert torch.equal(all_, one.repeat(rep))
    g = tr.refit_backward(torch.ones(rep * nt, device="cuda")).cpu().numpy().astype(np.float64)
    assert np.abs(g - rep * g1).max() <= 1e-9 * np.abs(g).max() or \
        np.all(np.abs(g - rep * g1) <= 2.0 ** -23 * np.abs(g) + 1e-9 * np.abs(g).max())

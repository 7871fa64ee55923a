"""Calls at the limits of a context, and what they leave for the next one."""
from __future__ import annotations

import os
import subprocess

import numpy as np
import pytest

from paper_2601_20569_gb300 import synth
from paper_2601_20569_gb300.options import TrackerOptions

pytestmark = pytest.mark.gpu

RX = synth.row_x()


def tracks(tr, dev):
    tr.track(*dev)
    return {k: v.cpu().numpy().copy() for k, v in tr.result().items()}


def same(a, b):
    return all(np.array_equal(a[k].view(np.uint8), b[k].view(np.uint8)) for k in a)


@pytest.mark.parametrize("graphs", [False, True])
@pytest.mark.parametrize("iters", [1, 2])
def test_tracklet_capacity_exceeded_then_a_valid_call(iters, graphs):
    """More start hits than tracklet slots, in the first sector-tracking iteration and
    (one slot short of both iterations' hits) in the second: the call reports the
    size it needs, and a call that fits gives a fresh context's tracks."""
    from paper_2601_20569_gb300 import tpc

    f = synth.generate("central_event", n_primaries=900, looper_frac=0.2, seed=21)
    s = synth.generate("one_sector", n_primaries=40)
    opts = TrackerOptions(seed_iters=iters)
    roomy = tpc.Tracker(RX, opts, mode=0, cap_clusters=f.n)
    dev = roomy.to_device(f.y, f.z, f.q, f.row, f.sector)
    sdev = roomy.to_device(s.y, s.z, s.q, s.row, s.sector)
    want = tracks(roomy, sdev)
    roomy.track(*dev)
    need = len(roomy.debug("starts"))
    first = int(roomy.debug("pass_start")[1]) if iters > 1 else need
    assert need >= first > 64 and (iters == 1 or need > first)
    roomy.close()
    for cap in {first - 1, need - 1, first // 3}:
        tr = tpc.Tracker(RX, opts, mode=0, cap_clusters=f.n, cap_tracklets=cap, use_graphs=graphs)
        for _ in range(3):
            with pytest.raises(tpc.TpcError) as e:
                tr.track(*dev)
            assert e.value.status == 3 and e.value.needed == (first if cap < first else need)
            assert same(tracks(tr, sdev), want)
        tr.close()


def run_with_internals(name, tmp_path, frame, opts):
    """Builds tests/cpp/<name>.cu, which includes a host source file of the library,
    against libtpc.so and runs it on a frame; returns the words it prints."""
    from paper_2601_20569_gb300 import build, tpc

    data = tmp_path / "frame.bin"
    with open(data, "wb") as out:
        np.array([frame.n, len(RX)], np.int64).tofile(out)
        out.write(bytes(tpc.make_options(opts, mode=0, cap_clusters=frame.n)))
        for a, dt in ((RX, np.float32), (frame.y, np.float32), (frame.z, np.float32),
                      (frame.row, np.uint8), (frame.sector, np.uint8)):
            np.ascontiguousarray(a, dtype=dt).tofile(out)
    exe = tmp_path / name
    here = os.path.dirname(os.path.abspath(__file__))
    subprocess.check_call([build._nvcc()] + build.COMMON +
                          [os.path.join(here, "cpp", name + ".cu"), "-o", str(exe), "-L" + build.HERE,
                           "-l:libtpc.so", "-Xlinker", "-rpath=" + build.HERE])
    r = subprocess.run([str(exe), str(data)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout.split()


def test_links_after_stale_bin_counts(tmp_path):
    f = synth.generate("one_sector")
    v = run_with_internals("links_scratch", tmp_path, f, TrackerOptions())
    assert v[0] == "links" and int(v[1]) > 0.5 * f.n
    assert v[2] == "changed" and int(v[3]) == 0


def test_call_after_an_interrupted_one(tmp_path):
    f = synth.generate("central_event", n_primaries=300, seed=8)
    v = run_with_internals("interrupted_call", tmp_path, f, TrackerOptions())
    assert v[0] == "tracks" and int(v[1]) > 100
    assert v[4] == "changed" and int(v[5]) == 0


REFIT_KEYS = ("cl_offset", "cl_ids", "params", "x", "sector")


def refit_setup(n_primaries=300, cap_clusters=None, **opts):
    import torch

    from paper_2601_20569_gb300 import tpc

    f = synth.generate("central_event", distort=True, n_primaries=n_primaries)
    tr = tpc.Tracker(RX, TrackerOptions(**opts), mode=0, cap_clusters=cap_clusters or f.n)
    coeff = torch.as_tensor(f.map).cuda()
    tr.set_map(coeff)
    dev = tr.to_device(f.y, f.z, f.q, f.row, f.sector)
    tr.track(*dev)
    return f, tr, dev, coeff, {k: tr.result()[k].clone() for k in REFIT_KEYS}


def first_tracks(t, n):
    refs = int(t["cl_offset"][n])
    return {"cl_offset": t["cl_offset"][:n + 1].clone(), "cl_ids": t["cl_ids"][:refs].clone(),
            **{k: t[k][:n].clone() for k in ("params", "x", "sector")}}


@pytest.mark.parametrize("row", [152, 159, 160, 255])
def test_refit_skips_a_track_with_a_row_that_does_not_exist(row):
    f, tr, dev, coeff, t = refit_setup()
    keys = ("chi2", "n_clusters", "params", "cov")
    want = {k: tr.refit(dev, t, coeff)[k].clone() for k in keys}
    nt = int(t["params"].shape[0])
    bad = nt // 2
    assert int(want["n_clusters"][bad]) > 0
    rows = dev[3].clone()
    o = int(t["cl_offset"][bad])
    ids = t["cl_ids"].clone()
    # (clusters may be shared by tracks: the bad one gets a copy of its own)
    c = int(ids[o + 3])
    more = [x if x is None else x.new_empty(x.shape[0] + 1) for x in dev]
    for a, b in zip(more, dev):
        a[:-1] = b
        a[-1] = b[c]
    more[3][:-1] = rows
    more[3][-1] = row
    ids[o + 3] = f.n
    got = tr.refit(tuple(more), dict(t, cl_ids=ids), coeff)
    assert int(got["n_clusters"][bad]) == 0 and float(got["chi2"][bad]) == 0.0
    keep = [i for i in range(nt) if i != bad and int(want["n_clusters"][i]) > 0]
    for k in keys:
        assert np.array_equal(got[k][keep].cpu().numpy().view(np.uint8),
                              want[k][keep].cpu().numpy().view(np.uint8)), k


def test_refit_without_room_for_its_map_leaves_the_last_one():
    """A refit refused for want of memory for its map (1.3 TB here; nothing is
    launched) does not touch the refit before it, which can still be
    differentiated: the gradient's FP64 sums differ by their order only."""
    import torch

    from paper_2601_20569_gb300 import tpc

    f, tr, dev, coeff, t = refit_setup()
    nt = int(t["params"].shape[0])
    w = torch.linspace(0.5, 1.5, nt, device="cuda")
    tr.refit(dev, t, coeff)
    want = tr.refit_backward(w).cpu().numpy()
    huge = coeff.new_zeros(1).expand(3, 20000, 2000, 2000)
    with pytest.raises(tpc.TpcError) as e:
        tr.refit(dev, first_tracks(t, nt // 3), huge)
    assert e.value.status == 5
    got = tr.refit_backward(w, tuple(coeff.shape)).cpu().numpy()
    assert np.abs(got - want).max() <= 2.0 ** -23 * np.abs(want).max()


def test_map_of_more_than_2_31_coefficients():
    """A constant map of 7.2e8 control points, read at its far end (every cluster of
    side A lies above its z range): the shift of a small constant map.  The spline
    weights sum to 1 within a few 2^-24, a correction of 0.25 cm to 1e-7 cm."""
    import torch

    f, tr, dev, coeff, t = refit_setup(n_primaries=100)
    side_a = torch.nonzero(t["sector"] < 18).flatten().cpu().numpy()
    assert len(side_a) > 20
    out = []
    for shape in ((2000, 2000, 180), (20, 16, 18)):
        c = torch.zeros((3,) + shape, device="cuda")
        c[2] = 0.25
        r = tr.refit(dev, t, c, z_range=(-1000.0, 1.0))
        out.append({k: r[k].cpu().numpy()[side_a].copy() for k in ("params", "n_clusters")})
        del c, r
    plain = tr.refit(dev, t, coeff.new_zeros(coeff.shape))["params"].cpu().numpy()[side_a]
    big, small = out
    fitted = (big["n_clusters"] > 0) & (big["n_clusters"] == small["n_clusters"])
    assert fitted.sum() > 0.9 * len(side_a)
    assert np.abs(np.median(big["params"][fitted, 1] - plain[fitted, 1]) - 0.25) < 0.01
    assert np.abs(big["params"] - small["params"])[fitted, 1].max() < 1e-3
    tr.close()
    torch.cuda.empty_cache()


def test_adjoint_takes_memory_for_its_tracks_only():
    """A context for up to 45,000 tracks, a refit of 200 of them: 200 step records of
    46 KB (in steps of 2 MB, rounded up to 256) and the gradient's partial sums (21 MB)."""
    import torch

    f, tr, dev, coeff, t = refit_setup(n_primaries=300, cap_clusters=1_650_000)
    few = first_tracks(t, 200)
    w = torch.ones(200, device="cuda")
    tr.refit(dev, few, coeff)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    tr.refit_backward(w)
    assert free - torch.cuda.mem_get_info()[0] < 64 << 20


@pytest.mark.parametrize("room", [700, 64])
def test_adjoint_in_the_memory_there_is(room):
    """33,000 tracks with room (MB) for a quarter of their step records, or hardly more
    than the gradient's partial sums: the gradient of the same refit with all of them
    (FP64 sums in another order)."""
    import torch

    f, tr, dev, coeff, t = refit_setup(n_primaries=1500, cap_clusters=3_500_000)
    nt, nr = int(t["params"].shape[0]), int(t["cl_ids"].shape[0])
    rep = -(-33000 // nt)
    many = {k: t[k].repeat((rep,) + (1,) * (t[k].dim() - 1)) for k in ("cl_ids", "params", "x", "sector")}
    step = torch.arange(rep, device="cuda", dtype=torch.int32)[:, None] * nr
    many["cl_offset"] = torch.cat([(t["cl_offset"][:-1] + step).reshape(-1),
                                   torch.tensor([rep * nr], device="cuda", dtype=torch.int32)])
    w = torch.linspace(0.5, 1.5, rep * nt, device="cuda")
    from paper_2601_20569_gb300 import tpc

    tight = tpc.Tracker(RX, TrackerOptions(), mode=0, cap_clusters=3_500_000)
    got = []
    for x in (tr, tight):
        x.refit(dev, many, coeff)
        hog = None
        if x is tight:  # (memory taken, not touched)
            torch.cuda.synchronize()
            torch.cuda.empty_cache()
            hog = torch.empty(torch.cuda.mem_get_info()[0] - (room << 20), dtype=torch.uint8, device="cuda")
        try:
            got.append(x.refit_backward(w).cpu().numpy().astype(np.float64))
        finally:
            del hog
            torch.cuda.empty_cache()
    assert np.abs(got[0] - got[1]).max() <= 2.0 ** -23 * np.abs(got[0]).max()


@pytest.mark.parametrize("ext", [0, 8])
def test_device_memory_of_a_context(ext):
    """What tpc.h states per cluster of capacity, and the candidates of the
    extrapolated rows; each of some hundred buffers rounded up to 2 MB at most."""
    import torch

    from paper_2601_20569_gb300 import tpc

    n = 40_000_000
    tpc.Tracker(RX, TrackerOptions(), mode=0, cap_clusters=1024).close()  # (loads the library)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    tr = tpc.Tracker(RX, TrackerOptions(ext_rows=ext), mode=0, cap_clusters=n)
    used = free - torch.cuda.mem_get_info()[0]
    tr.close()
    tracks = n / 40 + 4096
    per_ext_row = 2 * (8 * 8 + 4 + 1 + 2)  # candidates, chi2, assignment, count, sector
    assert used < 512 * n + ext * per_ext_row * tracks + (256 << 20)


@pytest.mark.parametrize("shape", [(20, 16, 18), (20, 24, 20)])  # sums in shared memory, in global
def test_adjoint_of_very_small_and_large_weights(shape):
    """The gradient is linear in the weights, and a power of two scales every float
    exactly: with weights outside the three-float sums' range (term by term in FP64)
    it is the scaled gradient, within one rounding to float and, where elements
    cancel, the FP64 sums' 2^-53 of the terms (at most 2^-40 of the largest)."""
    import torch

    f, tr, dev, coeff, t = refit_setup(n_primaries=400)
    coeff = torch.as_tensor(0.05 * np.random.default_rng(2).standard_normal((3,) + shape),
                            dtype=torch.float32).cuda()
    nt = int(t["params"].shape[0])
    w = torch.linspace(0.5, 1.5, nt, device="cuda")
    tr.refit(dev, t, coeff)
    want = tr.refit_backward(w).cpu().numpy().astype(np.float64)
    assert np.abs(want).max() > 1.0
    for k in (-70, 105):
        got = tr.refit_backward(w * 2.0 ** k).cpu().numpy().astype(np.float64) * 2.0 ** -k
        assert np.all(np.abs(got - want) <= 2.0 ** -23 * np.abs(want) + 2.0 ** -40 * np.abs(want).max())


def test_adjoints_of_two_contexts_on_two_threads():
    """Maps of 138 KB, 14 KB and 230 KB of accumulators (the last beyond shared
    memory) side by side: the attributes of the kernels belong to the process."""
    import threading

    import torch

    f, tr, dev, coeff, t = refit_setup(n_primaries=60)
    rng = np.random.default_rng(6)
    nt = int(t["params"].shape[0])
    failed = []
    torch.cuda.synchronize()

    def worker(shape):
        from paper_2601_20569_gb300 import tpc

        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                c = torch.as_tensor(0.02 * rng_maps[shape]).cuda()
                w = torch.ones(nt, device="cuda")
                x = tpc.Tracker(RX, TrackerOptions(), mode=0, cap_clusters=f.n)
                x.refit(dev, t, c)
                want = x.refit_backward(w).cpu().numpy()
                for _ in range(3000):
                    got = x.refit_backward(w).cpu().numpy()
                    if np.abs(got - want).max() > 2.0 ** -23 * np.abs(want).max():
                        failed.append((shape, "gradient"))
                x.close()
        except Exception as e:  # (reported by the test's own thread)
            failed.append((shape, repr(e)))

    shapes = [(20, 16, 18), (6, 6, 16), (20, 24, 20)]
    rng_maps = {s: rng.standard_normal((3,) + s).astype(np.float32) for s in shapes}
    threads = [threading.Thread(target=worker, args=(s,)) for s in shapes]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not failed, failed[:3]


@pytest.mark.parametrize("length", [1, 2, 15, 16, 17, 31, 32, 33, 48, 49, 64, 65, 100])
def test_adjoint_of_tracks_of_one_length(length):
    """The adjoint against the FP64 tape for tracks cut to one length, each with a norm
    of its own.  With clusters of 3 cm resolution the fit follows no cluster, so
    residuals stay near the map's random 0.2 cm at every length; the forward states
    round by up to 4 x 2^-24 x 250 cm per step, over 100 steps 10 times that: 6e-4 cm,
    below 5e-3 of the residuals."""
    import torch

    import oracle
    from paper_2601_20569_gb300 import tpc
    from tests.test_gpu_refit import device_tracks, host_tracks

    f, tr, dev, _, t = refit_setup(n_primaries=250)
    tr.close()
    dmap = (0.6 * np.random.default_rng(11).standard_normal((3, 20, 16, 18))).astype(np.float32)
    h = host_tracks(t)
    sel = np.nonzero(np.diff(h["offset"]) >= length)[0][:150]
    assert len(sel) > 30
    h = host_tracks(t, sel)
    ids = np.concatenate([h["ids"][o:o + length] for o in h["offset"][:-1]])
    h = dict(h, ids=ids, offset=np.arange(0, len(ids) + 1, length, dtype=np.int32))
    opts = TrackerOptions(sigma_y=3.0, sigma_z=3.0).as_dict()
    x = tpc.Tracker(RX, opts, mode=0, cap_clusters=f.n)
    w = np.random.default_rng(12).uniform(0.5, 1.5, len(sel))
    out = x.refit(dev, device_tracks(h), torch.as_tensor(dmap).cuda())
    r = oracle.refit(f.y, f.z, f.row, f.sector, RX, opts, h, dist_map=dmap, mode="f32")
    assert np.array_equal(out["n_clusters"].cpu().numpy(), r["rf_n"])
    assert (r["rf_n"] > 0).sum() > 0.8 * len(sel)
    g = x.refit_backward(torch.as_tensor(w, dtype=torch.float32).cuda()).cpu().numpy().ravel()
    tape = oracle.refit(f.y, f.z, f.row, f.sector, RX, opts, h, dist_map=dmap, frozen=r, weights=w,
                        mode="tape")["grad"]
    assert np.linalg.norm(tape) > 0
    assert np.linalg.norm(g - tape) < 5e-3 * np.linalg.norm(tape)
    x.close()


def test_refit_with_a_larger_map_between_replayed_graphs():
    """A refit whose map needs more room than the tracker's replaces the packed map
    that a captured chain reads: the chain is captured again."""
    import torch

    from paper_2601_20569_gb300 import tpc

    f = synth.generate("central_event", n_primaries=300, distort=True)
    rng = np.random.default_rng(9)
    small, large = (torch.as_tensor((0.05 * rng.standard_normal(s)).astype(np.float32)).cuda()
                    for s in ((3, 5, 6, 7), (3, 40, 30, 36)))
    tr = tpc.Tracker(RX, TrackerOptions(), mode=0, cap_clusters=f.n, use_graphs=True)
    tr.set_map(small)
    dev = tr.to_device(f.y, f.z, f.q, f.row, f.sector)
    want = tracks(tr, dev)
    assert same(tracks(tr, dev), want)
    t = {k: tr.result()[k].clone() for k in REFIT_KEYS}
    tr.refit(dev, t, large)
    hold = torch.full((1 << 20,), float("nan"), device="cuda")  # (the freed room's next user)
    assert same(tracks(tr, dev), want) and same(tracks(tr, dev), want)
    assert bool(torch.isnan(hold).all())

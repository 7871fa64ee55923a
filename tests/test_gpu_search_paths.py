"""The searches' dispatch by local density, and what one call leaves for the next:
neighbour links where a window's whole strips, its own bins or neither fit a mask;
removal tubes wider than a mask; a larger map after a smaller one under a captured
graph; a valid call after calls that failed at different stages."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2601_20569_gb300 import synth
from paper_2601_20569_gb300.options import TrackerOptions

pytestmark = pytest.mark.gpu

RX = synth.row_x()


def blob(k, dy, dz, span, seed):
    """k clusters per row in a dy x dz box on rows 40-46 of sector 4, and a few that
    stretch every row's z range to `span` (which sets the bins' size)."""
    rng = np.random.default_rng(seed)
    y, z, row = [], [], []
    for r in range(40, 47):
        y += list(rng.uniform(-dy / 2, dy / 2, k)) + [0.0, 0.0]
        z += list(60.0 + rng.uniform(0.0, dz, k)) + [60.0 - span / 2, 60.0 + span / 2]
        row += [r] * (k + 2)
    n = len(y)
    order = rng.permutation(n)
    return (np.array(y, np.float32)[order], np.array(z, np.float32)[order], np.zeros(n, np.uint16),
            np.array(row, np.uint8)[order], np.full(n, 4, np.uint8))


@pytest.mark.parametrize("k,dy,dz,span", [
    (1, 1, 1, 100), (12, 8, 8, 300), (31, 6, 6, 400), (32, 5, 5, 400), (33, 5, 5, 400),
    (60, 30, 5, 400), (60, 6, 6, 400), (150, 30, 20, 200), (900, 30, 30, 30)])
def test_links_at_every_density(k, dy, dz, span):
    from paper_2601_20569_gb300 import tpc

    y, z, q, row, sec = blob(k, dy, dz, span, k)
    opts = TrackerOptions(brute_force=1).as_dict()
    ref = oracle.track(y, z, row, sec, RX, opts)
    for fast in (0, 1):
        tr = tpc.Tracker(RX, opts, mode=fast, cap_clusters=max(len(y), 1024),
                         cap_tracklets=len(y) + 64)
        tr.track(*tr.to_device(y, z, q, row, sec))
        sid, lup, ldn = tr.debug("sid"), tr.debug("lup"), tr.debug("ldn")
        tr.close()
        if fast:  # (contracted sums may part equal distances: the links exist alike)
            assert np.array_equal(np.sort(sid[lup >= 0]), np.nonzero(ref["link_up"] >= 0)[0])
            continue
        for name, got in (("link_up", lup), ("link_dn", ldn)):
            ids = np.full(len(y), -1, np.int64)
            ids[sid] = np.where(got >= 0, sid[np.maximum(got, 0)], -1)
            assert np.array_equal(ids, ref[name]), name


@pytest.mark.parametrize("widths", [(1.5, 0.75, 2.0), (9.0, 0.0, 12.0), (0.4, 20.0, 1.0)])
def test_removal_tubes_of_any_width(widths):
    from paper_2601_20569_gb300 import tpc

    f = synth.generate("central_event", n_primaries=1200, looper_frac=0.2, seed=77)
    opts = TrackerOptions(cr_mode=2, cr_protect=widths[0], cr_remove=widths[1],
                          cr_occ_w=widths[2]).as_dict()
    tr = tpc.Tracker(RX, opts, mode=0, cap_clusters=f.n)
    tr.track(*tr.to_device(f.y, f.z, f.q, f.row, f.sector))
    flags = tr.cluster_removal(opts)["flags"].cpu().numpy().astype(np.int32)
    ref = oracle.track(f.y, f.z, f.row, f.sector, RX, opts, full=True)
    assert np.array_equal(flags, ref["cr_flags"])


def tracks(tr, dev):
    tr.track(*dev)
    return {k: v.cpu().numpy().copy() for k, v in tr.result().items()}


def same(a, b):
    return all(np.array_equal(a[k].view(np.uint8), b[k].view(np.uint8)) for k in a)


@pytest.mark.parametrize("graphs", [False, True])
def test_map_grows_under_a_graph(graphs):
    import torch

    from paper_2601_20569_gb300 import tpc

    f = synth.generate("central_event", n_primaries=500, distort=True)
    rng = np.random.default_rng(5)
    small = torch.as_tensor((0.05 * rng.standard_normal((3, 5, 6, 7))).astype(np.float32)).cuda()
    large = torch.as_tensor(f.map).cuda()
    tr = tpc.Tracker(RX, TrackerOptions(), mode=0, cap_clusters=f.n, use_graphs=graphs)
    dev = tr.to_device(f.y, f.z, f.q, f.row, f.sector)
    got = []
    for coeff in (small, large, small, None, large):
        tr.set_map(coeff)
        got.append((tracks(tr, dev), tracks(tr, dev)))
        fresh = tpc.Tracker(RX, TrackerOptions(), mode=0, cap_clusters=f.n)
        if coeff is not None:
            fresh.set_map(coeff)
        want = tracks(fresh, dev)
        fresh.close()
        assert same(got[-1][0], want) and same(got[-1][1], want)
    # new values in the same tensor are those of the next call
    large.mul_(0.5)
    changed = tracks(tr, dev)
    assert not same(changed, got[-1][0])
    large.mul_(2.0)
    assert same(tracks(tr, dev), got[-1][0])


@pytest.mark.parametrize("graphs", [False, True])
def test_valid_call_after_failed_ones(graphs):
    from paper_2601_20569_gb300 import tpc

    f = synth.generate("central_event", n_primaries=700, seed=3)
    fresh = tpc.Tracker(RX, TrackerOptions(), mode=0, cap_clusters=f.n)
    dev = fresh.to_device(f.y, f.z, f.q, f.row, f.sector)
    want = tracks(fresh, dev)
    tr = tpc.Tracker(RX, TrackerOptions(), mode=0, cap_clusters=f.n, use_graphs=graphs)
    nan = f.y.copy()
    nan[f.n // 2] = np.nan
    far = f.sector.copy()
    far[5] = 77
    pile_y, pile_z = f.y.copy(), f.z.copy()
    pile = (f.row >= 25) & (f.row < 35)
    pile_y[pile], pile_z[pile] = 1.0, 20.0
    rows = np.where(pile, 30, f.row).astype(np.uint8)
    one = np.where(pile, 2, f.sector).astype(np.uint8)
    assert pile.sum() > 1024
    for bad in ((nan, f.z, f.q, f.row, f.sector), (f.y, f.z, f.q, f.row, far),
                (pile_y, pile_z, f.q, rows, one)):
        with pytest.raises(tpc.TpcError):
            tr.track(*tr.to_device(*bad))
        assert same(tracks(tr, dev), want)
    few = tpc.Tracker(RX, TrackerOptions(), mode=0, cap_clusters=f.n, cap_tracks=100,
                      use_graphs=graphs)
    small = synth.generate("one_sector", n_primaries=40)
    sdev = few.to_device(small.y, small.z, small.q, small.row, small.sector)
    ok = tracks(few, sdev)
    with pytest.raises(tpc.TpcError):
        few.track(*dev)  # more merged tracks than the context holds
    assert same(tracks(few, sdev), ok)

"""The block-wide walk of the seeding kernel at its edges.

Pairs are walked in groups of 32 and blocks of 12 or 24 groups per warp, triplets
wait in queues of 128 per warp, UV combinations go in blocks of 1024.  Batches
of up to four items per SM run in larger CTAs or with more registers, and so do
those of more than five and up to eight, in two rounds.  Wide third-hit bands and
windows, tiny events and batch sizes around these limits reach every branch; the
oracle, and the same batch in CTAs of other sizes, say what is right."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import parity  # noqa: E402
from conftest import workload  # noqa: E402
from paper_2606_14480_gb300 import st  # noqa: E402
from synth import calibrate_zmatch, make_events  # noqa: E402
from test_gpu_parity import run_gpu  # noqa: E402

KEYS = ("ev_off", "hits", "params", "state", "n_hits", "status", "velo_idx", "chi2", "n_long")


@pytest.fixture(scope="module")
def zmx():
    return calibrate_zmatch(7826.0)


def run(b, zmx, **over):
    _, gcfg = parity.config_pair(zmx, **over)
    ctx = st.Context(gcfg)
    out = st.run_batch(ctx, st.DeviceBatch.from_synth(b)).to_numpy()
    ctx.close()
    return out


@pytest.mark.parametrize("n,tracks,over", [
    (6, 400, dict(m_lo=0.0, m_hi=40.0, cand_cap=65536)),                     # queues of triplets run over
    (2, 200, dict(m_lo=0.0, m_hi=400.0, chi2x_max=0.5, cand_cap=65536)),     # single groups hold more than a queue
    (6, 300, dict(uv_y_overlap=2500.0, n_uv_min=3)),                         # blocks of UV combinations
    (40, 1, {}), (40, 3, dict(n_uv_min=2)),                                  # less than a warp of anything
])
def test_walk_edges_parity_and_shapes(n, tracks, over, zmx):
    b = make_events(n, seed=4001, tracks=("fixed", tracks))
    ocfg, gcfg = parity.config_pair(zmx, **over)
    gpu, _ = run_gpu(b, gcfg)
    assert (gpu["status"] == 0).all()
    # the harness's bars, except that on chi2: wide bands make combinations
    # whose chi2 is far below the default band's, where its relative error says
    # nothing about the walk
    rep = parity.compare_seeding(gpu, ocfg, b)
    assert rep.agreement >= parity.AGREE_MIN and not rep.untraced and not rep.bad_params, rep.summary()
    for shape in (dict(threads_seed=64), dict(threads_seed=96, ctas_per_sm=1), dict(threads_seed=256, ctas_per_sm=8)):
        other = run(b, zmx, **over, **shape)
        for k in ("ev_off", "hits", "params", "state"):
            assert np.array_equal(other[k], gpu[k]), (shape, k)


@pytest.mark.parametrize("over", [
    dict(iter_layers=[[0, 4, 11], [11, 7, 3], [0, 7, 11]]),  # the second iteration's windows are empty
    dict(iter_layers=[[11, 7, 3], [0, 4, 11], [0, 7, 11]]),  # the first one's
    dict(iter_layers=[[0, 4, 11], [11, 7, 3], [0, 7, 11]], n_iter=3),
    dict(dx3_scale=-1.0),                                     # all of them
])
def test_empty_two_hit_windows(over, zmx):
    """Two-hit windows that end before they start hold no hit and take nothing
    from the other iterations'."""
    b = make_events(6, seed=4031, tracks=("fixed", 60))
    ocfg, gcfg = parity.config_pair(zmx, **over)
    gpu, cnt = run_gpu(b, gcfg)
    assert (gpu["status"] == 0).all()
    rep = parity.compare_seeding(gpu, ocfg, b)
    assert rep.agreement >= parity.AGREE_MIN and not rep.untraced and not rep.bad_params, rep.summary()
    none = "dx3_scale" in over
    assert (gpu["ev_off"][-1] == 0) == none and (cnt["pairs"] == 0) == none


@pytest.mark.parametrize("items", [2, 3, 4, 5, 8, 10])
@pytest.mark.parametrize("mode", [{}, dict(uv_mode=1), dict(iter_mode=1)], ids=["hlt1", "hough", "seq"])
def test_larger_ctas_give_the_same(mode, items, zmx):
    """Around the batch sizes (items per SM) at which another kind of CTAs
    begins, and one that the configured CTAs take either way: every event's
    result is that of the batch one event larger."""
    sms = items * torch.cuda.get_device_properties(0).multi_processor_count // 2
    b = workload("run3", n_events=sms + 1)
    big = run(b, zmx, **mode)
    small = run(b.subset(range(sms)), zmx, **mode)
    n = small["ev_off"][-1]
    assert np.array_equal(small["ev_off"], big["ev_off"][:-1]) and (big["status"] == 0).all()
    for k in KEYS[1:]:
        assert np.array_equal(small[k], big[k][:len(small[k])]), k
    assert n > 0


@pytest.mark.parametrize("mode", [{}, dict(uv_mode=1), dict(iter_mode=1)], ids=["hlt1", "hough", "seq"])
def test_two_rounds_of_wider_ctas(mode, zmx):
    """Between five and eight items per SM: the CTAs with more registers take
    the items from the queue in cost order, and in a graph leave the last
    events' matching to each other.  The results are those of the configured
    CTAs (a set ctas_per_sm)."""
    n = 13 * torch.cuda.get_device_properties(0).multi_processor_count // 4
    b = workload("run3", n_events=n)
    want = run(b, zmx, ctas_per_sm=5, **mode)
    got = run(b, zmx, **mode)
    _, gcfg = parity.config_pair(zmx, **mode)
    ctx = st.Context(gcfg)
    db = st.DeviceBatch.from_synth(b)
    out = st.DeviceOutputs(n, max(1024, b.n_hits // 4))
    gr = ctx.st_graph_create(db.hits, db.velo_s, out.seeds, out.long)
    gr.st_graph_launch()
    gr.st_graph_launch()
    torch.cuda.synchronize()
    graph = out.to_numpy()
    gr.close()
    ctx.close()
    assert (want["status"] == 0).all() and want["ev_off"][-1] > 100 * n
    for k in KEYS:
        assert np.array_equal(want[k], got[k]) and np.array_equal(want[k], graph[k]), k


def _concat(parts):
    """One batch of (events, hits kept of each or None) pairs."""
    x, zone, velo, eo, vo = [], [], [], [0], [0]
    for b, keep in parts:
        for e in range(b.n_events):
            h0, h1 = int(b.ev_off[e]), int(b.ev_off[e + 1])
            h1 = h1 if keep is None else h0 + keep
            assert h1 <= b.ev_off[e + 1]
            x.append(b.x[h0:h1])
            zone.append(b.zone[h0:h1])
            velo.append(b.velo[b.velo_off[e]:b.velo_off[e + 1]])
            eo.append(eo[-1] + h1 - h0)
            vo.append(vo[-1] + len(velo[-1]))
    return np.array(eo), np.concatenate(x), np.concatenate(zone), np.array(vo), np.concatenate(velo)


@pytest.mark.parametrize("mode", [{}, dict(uv_mode=1), dict(iter_mode=1)], ids=["hlt1", "hough", "seq"])
def test_large_events_beside_ordinary(mode, zmx):
    """Batches that may hold large events: those events' containers and items
    run in larger CTAs beside the others.  Around the sizes that divide them,
    with a faulty large event and one above the bound, the results are those of
    the launches without the division (a set ctas_per_sm)."""
    d = make_events(2, seed=4021, tracks=("fixed", 500))
    g = make_events(1, seed=4022, tracks=("fixed", 1300))
    assert np.diff(d.ev_off).min() > 6144 and np.diff(g.ev_off).min() > 16385
    s = make_events(130, seed=4023, tracks=("fixed", 25))
    eo, x, zone, vo, velo = _concat([(s, None), (d, 4096), (s.subset(range(9)), 0), (d, 4097), (d, None), (g, 16384),
                                     (d, 6144), (g, 16385), (d, None), (s, None)])
    last = 130 + 2 + 9 + 2 + 2 + 1 + 2 + 1  # the first of the two large events after the 16385-hit one
    zone = zone.copy()
    zone[eo[last] + 5000] = 24
    cap = 80 * (len(eo) - 1)
    for mh in (16385, 16384):
        res = []
        for shape in (dict(ctas_per_sm=8), {}):
            _, gcfg = parity.config_pair(zmx, cand_cap=16384, **mode, **shape)
            db = st.DeviceBatch(eo, x, zone, vo, velo, max_hits=mh)
            ctx = st.Context(gcfg)
            res.append(st.run_batch(ctx, db, cap=cap).to_numpy())
            if not mode and not shape:
                out = st.DeviceOutputs(len(eo) - 1, cap)
                gr = ctx.st_graph_create(db.hits, db.velo_s, out.seeds, out.long)
                gr.st_graph_launch()
                gr.st_graph_launch()
                torch.cuda.synchronize()
                res.append(out.to_numpy())
                gr.close()
            ctx.close()
        want = np.zeros(len(eo) - 1, np.int32)
        want[last] = st.ST_EINVAL
        want[np.diff(eo) > mh] = st.ST_OVERFLOW
        for r in res:
            # (the HLT2-style mode stores all UV combinations of an item and
            # refuses those whose store runs over)
            full = (r["status"] == st.ST_OVERFLOW) & (np.diff(eo) > 6144) if mode.get("iter_mode") else False
            assert np.array_equal(r["status"], np.where(full, st.ST_OVERFLOW, want))
            assert r["ev_off"][-1] > 1000
            for k in KEYS:
                assert np.array_equal(r[k], res[0][k]), (mh, k)


def test_large_events_in_a_callers_capture(zmx):
    """A batch that may hold large events, captured by the caller: the work on
    the context's own stream becomes part of the caller's graph."""
    s = make_events(200, seed=4024, tracks=("fixed", 30))
    d = make_events(2, seed=4025, tracks=("fixed", 500))
    eo, x, zone, vo, velo = _concat([(s, None), (d, None)])
    n = len(eo) - 1
    _, gcfg = parity.config_pair(zmx)
    db = st.DeviceBatch(eo, x, zone, vo, velo)
    assert db.max_hits > 6144
    cap = 80 * n
    ctx = st.Context(gcfg)
    want = st.run_batch(ctx, db, cap=cap).to_numpy()
    out = st.DeviceOutputs(n, cap)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ctx.seeding_run(db.hits, out.seeds)
        ctx.matching_run(db.velo_s, out.seeds, out.long)
    for _ in range(2):
        for a in (out.hits, out.velo_idx, out.n_long):
            a.fill_(-7)
        g.replay()
        torch.cuda.synchronize()
        got = out.to_numpy()
        for k in KEYS:
            assert np.array_equal(got[k], want[k]), k
    del g
    again = st.run_batch(ctx, db, cap=cap).to_numpy()
    assert np.array_equal(again["hits"], want["hits"]) and want["ev_off"][-1] > 1000
    ctx.close()


@pytest.mark.parametrize("n,tracks,over", [
    (60, 150, {}),                                       # one CTA per item
    (20, 260, {}),                                       # halves with more hits than shared memory holds
    (48, 60, dict(m_lo=0.0, m_hi=40.0, chi2x_max=1e9)),  # more candidates than the first step's scratch holds
    (48, 60, dict(uv_tol=40.0, n_uv_min=2)),             # more UV combinations than it holds
    (48, 60, dict(iter_mode=1, uv_tol=40.0, n_uv_min=2)),
    (48, 60, dict(uv_mode=1, uv_tol=10.0)),              # Hough hypotheses: more valid ones than it holds
])
def test_static_entry_in_two_steps(n, tracks, over, zmx):
    """seeding_run_static runs the items with little scratch each first and
    again, with all they may need, those that ask for more."""
    b = make_events(n, seed=4011, tracks=("fixed", tracks))
    _, gcfg = parity.config_pair(zmx, **over)
    ctx = st.Context(gcfg)
    db = st.DeviceBatch.from_synth(b)
    cap = max(1024, b.n_hits // 4)
    ref, out = st.DeviceOutputs(n, cap), st.DeviceOutputs(n, cap)
    ctx.seeding_run(db.hits, ref.seeds)
    rc, msg = st.seeding_run_static(gcfg, db.hits, out.seeds)
    assert rc == st.ST_OK, msg
    r, g = ref.to_numpy(), out.to_numpy()
    for k in ("ev_off", "hits", "params", "state", "n_hits", "status"):
        assert np.array_equal(r[k], g[k]), k
    ctx.close()

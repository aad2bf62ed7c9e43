"""Matching and UT search at the edges of their layouts: VELO segments in
chunks of 512 and off 16-byte alignment, larger CTAs for small batches, UT hits
around what shared memory holds and batches of several rounds."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle  # noqa: E402
import parity  # noqa: E402
from conftest import workload  # noqa: E402
from paper_2606_14480_gb300 import st  # noqa: E402
from synth import calibrate_zmatch, ghost_nn_weights, make_events  # noqa: E402


@pytest.fixture(scope="module")
def zmx():
    return calibrate_zmatch(7826.0)


@pytest.mark.parametrize("mode", [{}, dict(velo_unique=1), dict(final_sel=1)], ids=["plain", "unique", "final"])
def test_match_layouts(mode, zmx):
    """Chunk edges, an unaligned VELO array and other CTA shapes: the same pairs."""
    counts = [0, 1, 64, 511, 512, 513, 1024, 1100]
    b = make_events(len(counts), seed=4101, tracks=("fixed", 150))
    rng = np.random.default_rng(4102)
    velo = np.concatenate([b.velo[rng.integers(0, len(b.velo), n)] * np.float32(1 if n < 65 else 1.0001)
                           for n in counts]).astype(np.float32)
    for e, n in enumerate(counts):  # each event's own segments first
        o, k = sum(counts[:e]), min(n, int(b.velo_off[e + 1] - b.velo_off[e]))
        velo[o:o + k] = b.velo[b.velo_off[e]:b.velo_off[e] + k]
    vo = np.concatenate([[0], np.cumsum(counts)])
    db = st.DeviceBatch(b.ev_off, b.x, b.zone, vo, velo)
    ref = None
    for shape in ({}, dict(ctas_per_sm=1), dict(threads_match=64, ctas_per_sm=8), dict(threads_match=512)):
        for shift in (0, 1):
            flat = torch.zeros(4 * len(velo) + 1, device="cuda")
            flat[shift:shift + 4 * len(velo)] = torch.as_tensor(velo.reshape(-1), device="cuda")
            v = st.StVelo(len(counts), db.velo_s.ev_off, flat.data_ptr() + 4 * shift)
            _, gcfg = parity.config_pair(zmx, **mode, **shape)
            ctx = st.Context(gcfg)
            if mode.get("final_sel"):
                ctx.st_set_ghost_nn(ghost_nn_weights())
            out = st.DeviceOutputs(len(counts), 8192)
            ctx.seeding_run(db.hits, out.seeds)
            ctx.matching_run(v, out.seeds, out.long)
            r = out.to_numpy()
            ctx.close()
            n = int(r["ev_off"][-1])
            for e in range(len(counts)):
                idx = r["velo_idx"][r["ev_off"][e]:r["ev_off"][e + 1]]
                assert r["n_long"][e] == (idx >= 0).sum() and (idx < counts[e]).all()
            keys = ("velo_idx", "chi2") + (("ghost_prob",) if mode.get("final_sel") else ())
            got = [r[k][:n] for k in keys] + [r["n_long"]]
            if ref is None:
                ref = got
                assert r["n_long"][3:].min() > 0
            for a, c in zip(ref, got):
                assert np.array_equal(a, c), (shape, shift)


@pytest.mark.parametrize("per_sm", [4, 6, 15])
@pytest.mark.parametrize("mode", [{}, dict(velo_unique=1)], ids=["plain", "unique"])
def test_match_rounds(mode, per_sm, zmx):
    """On both sides of the batch sizes at which the matching takes CTAs with
    fewer registers: the pairs are those of the configured CTAs."""
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    b = make_events(n + 1, seed=4104, tracks=("fixed", 12))
    for k in (n, n + 1):
        db = st.DeviceBatch.from_synth(b.subset(range(k)))
        res = []
        for shape in (dict(ctas_per_sm=8), {}):
            _, gcfg = parity.config_pair(zmx, **mode, **shape)
            ctx = st.Context(gcfg)
            res.append(st.run_batch(ctx, db).to_numpy())
            ctx.close()
        assert res[0]["n_long"].sum() > k
        for key in ("velo_idx", "chi2", "n_long"):
            assert np.array_equal(res[0][key], res[1][key]), (k, key)


@pytest.mark.parametrize("nu", [0, 1, 767, 768, 769, 4096, 4097])
def test_ut_sizes(nu, zmx):
    """UT hits of an event around the threads' shares and shared memory."""
    b = workload("run3", n_events=6)
    ocfg, gcfg = parity.config_pair(zmx)
    rng = np.random.default_rng(4103)
    ux, ul = [], []
    for e in range(b.n_events):
        x, l = b.ut_of(e)
        more = max(nu - len(x), 0)
        ux.append(np.concatenate([x, rng.uniform(-1500, 1500, more).astype(np.float32)])[:nu])
        ul.append(np.concatenate([l, rng.integers(0, 4, more).astype(np.int32)])[:nu])
    db = st.DeviceBatch(b.ev_off, b.x, b.zone, b.velo_off, b.velo)
    db.add_ut(np.arange(b.n_events + 1) * nu, np.concatenate(ux), np.concatenate(ul))
    ctx = st.Context(gcfg)
    out = st.run_batch(ctx, db)
    pre = out.velo_idx.cpu().numpy().copy()
    ctx.ut_run(db.velo_s, out.seeds, db.ut, out.long, out.ut_out)
    r = out.to_numpy()
    ctx.close()
    for e in range(b.n_events):
        s0, s1 = int(r["ev_off"][e]), int(r["ev_off"][e + 1])
        w = oracle.ut_search(ocfg, b.velo_of(e), r["state"][s0:s1], pre[s0:s1], ux[e], ul[e], ledger_tau=1e-4)
        led = w["ledger"]
        near = {int(h[0]) for h in led[led["margin"] <= parity.TAU]["hits"]} if len(led) else set()
        for k in range(s1 - s0):
            if pre[s0 + k] >= 0 and k not in near:
                assert np.array_equal(r["ut_hits"][s0 + k], w["ut_hits"][k]), (e, k)
                assert r["velo_idx"][s0 + k] == w["velo_idx"][k]


def test_ut_rounds(zmx):
    """More events than CTAs at once: each event's hits are those it gets in a
    small batch."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    one = workload("run3", n_events=40)
    reps = (8 * sms + 3) // 40 + 2
    _, gcfg = parity.config_pair(zmx)
    res = []
    for n in (1, reps):
        db = st.DeviceBatch(*[np.concatenate([[0]] + [o[1:] + k * o[-1] for k in range(n)]) if i in (0, 3) else
                              np.concatenate([o] * n) for i, o in
                              enumerate((one.ev_off, one.x, one.zone, one.velo_off, one.velo))])
        db.add_ut(np.concatenate([[0]] + [one.ut_off[1:] + k * one.ut_off[-1] for k in range(n)]),
                  np.concatenate([one.ut_x] * n), np.concatenate([one.ut_layer] * n))
        ctx = st.Context(gcfg)
        out = st.run_batch(ctx, db)
        ctx.ut_run(db.velo_s, out.seeds, db.ut, out.long, out.ut_out)
        res.append(out.to_numpy())
        ctx.close()
    a, b = res
    n = int(a["ev_off"][-1])
    assert n > 0 and int(b["ev_off"][-1]) == n * reps
    for k in ("ut_hits", "ut_n", "ut_gamma", "velo_idx", "chi2"):
        for q in range(reps):
            assert np.array_equal(b[k][q * n:(q + 1) * n], a[k][:n]), (k, q)
    assert np.array_equal(b["n_long"], np.tile(a["n_long"], reps))

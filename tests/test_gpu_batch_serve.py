"""Batched and served plotting give every plot exactly the tables it gets
alone (the oracle's), whatever the mix of K and keys."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import oracle as orc  # noqa: E402
from paper_2606_14007_gb300.inputs import plot_key  # noqa: E402


@pytest.fixture(scope="module")
def vx():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_14007_gb300 import vaultx
    return vaultx


_cache = {}


def oracle_tables(K, seed):
    if (K, seed) not in _cache:
        key = plot_key(seed)
        t1 = orc.table1(K, key)
        _cache[(K, seed)] = (t1, orc.match(key, t1, orc.default_distance(K)))
    return _cache[(K, seed)]


def copy_table(vx, h, which):
    _, n, rb, _ = vx.vx_table_info(h, which)
    host = torch.empty(max(1, n * rb), dtype=torch.uint8).pin_memory()
    vx.vx_table_copy(h, which, host.data_ptr(), n * rb)
    torch.cuda.synchronize()
    return host[: n * rb].numpy().reshape(n, rb)


@pytest.mark.parametrize("placement", [1, 2], ids=["lookback", "slots"])
def test_batch_mixed_k_equals_oracle(vx, placement):
    mix = [(10, 101), (14, 102), (16, 103), (18, 104), (20, 105), (12, 106), (22, 107), (17, 108),
           (1, 109), (24, 110)]
    plots = [vx.Plot(K, plot_key(s), vx.make_opts(t2_placement=placement)) for K, s in mix]
    handles = [p.handle for p in plots]
    for rep in range(2):  # the second launch replays the recorded graph
        vx.vx_plot_batch(handles)
        for (K, s), p in zip(mix, plots):
            p.sync()
            if K > 22:
                continue
            r1, r2 = oracle_tables(K, s)
            assert np.array_equal(p.t1.cpu().numpy(), r1), (rep, K)
            assert np.array_equal(p.t2.cpu().numpy(), r2), (rep, K)
    # the K=24 member equals its own single-plot run
    single = vx.Plot(24, plot_key(110))
    single.run()
    single.sync()
    assert torch.equal(single.t1, plots[-1].t1) and torch.equal(single.t2, plots[-1].t2)
    for p in plots + [single]:
        p.close()


def test_serve_mix_equals_oracle(vx):
    srv = vx.vx_serve_create()
    rng = np.random.default_rng(9)
    reqs = []
    for r in range(16):
        K = int(rng.integers(12, 21))
        seed = 500 + r
        reqs.append((vx.vx_serve_submit(srv, K, plot_key(seed)), K, seed))
        if r % 5 == 4:
            vx.vx_serve_step(srv)   # later requests arrive while earlier ones run
    done = {}
    t0 = time.time()
    while len(done) < len(reqs):
        assert time.time() - t0 < 120, "server did not finish"
        for t, K, seed in reqs:
            if t in done:
                continue
            st, h = vx.vx_serve_poll(srv, t)
            assert st != vx.VX_FAILED
            if st == vx.VX_DONE:
                done[t] = h
        time.sleep(0.002)
    for t, K, seed in reqs:
        h = done[t]
        r1, r2 = oracle_tables(K, seed)
        assert np.array_equal(copy_table(vx, h, vx.VX_TABLE1), r1)
        assert np.array_equal(copy_table(vx, h, vx.VX_TABLE2), r2)
        assert vx.vx_serve_latency(srv, t) > 0
        vx.vx_plot_destroy(h)
    assert vx.vx_serve_step(srv) == 0
    vx.vx_serve_destroy(srv)


def test_serve_rejects_oversized(vx):
    srv = vx.vx_serve_create(vx.vx_serve_opts(size=0, memory_budget=1 << 20))
    with pytest.raises(vx.VxError):
        vx.vx_serve_submit(srv, 20, plot_key(1))
    vx.vx_serve_destroy(srv)


def test_batch_mixed_scope_and_placement(vx):
    # One batch launch mixing cross-bucket and bucket-scope plots (the
    # halo-capable kernel instances run both kinds) and both Table-2
    # placements (a mixed launch places every plot by look-back): each plot
    # equals its own oracle.
    mix = [(14, 120, dict(match_scope=1)), (16, 121, dict(t2_placement=1, nonces_per_thread=16)),
           (18, 122, dict(match_scope=1, t2_placement=2)),
           (12, 123, dict(t2_placement=2)), (20, 124, dict(match_scope=1)), (1, 125, dict(match_scope=1))]
    plots = [vx.Plot(K, plot_key(s), vx.make_opts(**kw)) for K, s, kw in mix]
    for rep in range(2):
        vx.vx_plot_batch([p.handle for p in plots])
        for (K, s, kw), p in zip(mix, plots):
            p.sync()
            key = plot_key(s)
            t1 = orc.table1(K, key)
            D = orc.default_distance(K)
            r2 = orc.match_global(key, t1, D) if kw.get("match_scope") else orc.match(key, t1, D)
            assert np.array_equal(p.t1.cpu().numpy(), t1), (rep, K)
            assert np.array_equal(p.t2.cpu().numpy(), r2), (rep, K)
    for p in plots:
        p.close()


@pytest.mark.parametrize("placement", [0, 1], ids=["slots", "lookback"])
def test_batch_results_of_good_and_failed_plots(vx, placement):
    # each plot's status and counts after a batch, for the plots whose results
    # the last kernel leaves in pinned memory and for the others: a Table 2
    # that is too small, one that fits, a slot overflow; then the match alone
    # on a larger buffer, a run of its own between two batches
    opts = [dict(t2_capacity=16), dict(), dict(partition_log2=6, slack_sigma=1)]
    mix = [(16, 201), (14, 202), (18, 203)]
    plots = [vx.Plot(K, plot_key(s), vx.make_opts(t2_placement=placement, **o)) for (K, s), o in zip(mix, opts)]
    handles = [p.handle for p in plots]
    want = [oracle_tables(K, s)[1] for K, s in mix]
    for rep in range(2):
        vx.vx_plot_batch(handles)
        codes = [vx.vx_sync(h, check=False) for h in handles]
        assert codes == [vx.VX_ENOMEM, vx.VX_OK, vx.VX_EOVERFLOW], (rep, codes)
        assert vx.vx_table_info(handles[0], vx.VX_TABLE2, check=False)[1] == want[0].shape[0]
        assert vx.vx_table_info(handles[1], vx.VX_TABLE2)[1] == want[1].shape[0]
        plots[1].run()
        assert plots[1].sync() == want[1].shape[0]
        assert np.array_equal(plots[1].t2.cpu().numpy(), want[1])
    vx.vx_plot_batch(handles)
    need = want[0].shape[0]
    big = torch.empty(16 * need + 256, dtype=torch.uint8, device="cuda")
    p = plots[0]
    vx.vx_plot_bind(p.handle, p._t1.data_ptr(), big.data_ptr(), p._scratch.data_ptr(), need)
    vx.vx_match(p.handle)
    assert vx.vx_sync(p.handle) == vx.VX_OK
    assert np.array_equal(big[: 16 * need].view(need, 16).cpu().numpy(), want[0])
    torch.cuda.synchronize()
    for p in plots:
        p.close()


@pytest.mark.parametrize("placement", [0, 1], ids=["slots", "lookback"])
def test_batch_follows_rebound_tables(vx, placement):
    # The same handles batched again after a plot's Table 2, then its Table 1,
    # was bound elsewhere with the scratch kept: the batch fills the new
    # buffers, up to the new capacity, and leaves the old ones alone.
    opts = [dict(t2_capacity=16), dict()]
    mix = [(16, 211), (14, 212)]
    plots = [vx.Plot(K, plot_key(s), vx.make_opts(t2_placement=placement, **o)) for (K, s), o in zip(mix, opts)]
    handles = [p.handle for p in plots]
    r1, r2 = oracle_tables(*mix[0])
    need, p = r2.shape[0], plots[0]
    vx.vx_plot_batch(handles)
    assert vx.vx_sync(p.handle, check=False) == vx.VX_ENOMEM
    big = torch.zeros(16 * need + 256, dtype=torch.uint8, device="cuda")
    t1 = torch.zeros_like(p._t1)
    for table1 in (p._t1, t1):
        vx.vx_plot_bind(p.handle, table1.data_ptr(), big.data_ptr(), p._scratch.data_ptr(), need)
        p._t2.zero_()
        big.zero_()
        table1.zero_()
        vx.vx_plot_batch(handles)
        assert [vx.vx_sync(h, check=False) for h in handles] == [vx.VX_OK, vx.VX_OK]
        assert vx.vx_table_info(p.handle, vx.VX_TABLE2)[1] == need
        assert np.array_equal(big[: 16 * need].view(need, 16).cpu().numpy(), r2)
        assert np.array_equal(table1[: r1.size].view(-1, 12).cpu().numpy(), r1)
        assert int(p._t2.max()) == 0
    for p in plots:
        p.close()

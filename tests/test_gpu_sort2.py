"""Table 2 sorted by hash2 (vx_sort_table2) against the oracle's sort of the
oracle's Table 2, byte for byte, through the C ABI."""
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


def sorted_plot(vx, K, key, kw, split=False):
    p = vx.Plot(K, key, vx.make_opts(**kw) if kw else None)
    p.run_split() if split else p.run()
    n2 = p.sync()
    wb = vx.vx_sort_table2_work_bytes(p.handle)
    work = torch.empty(max(wb, 256), dtype=torch.uint8, device="cuda")
    vx.vx_sort_table2(p.handle, work.data_ptr(), wb)
    assert vx.vx_sync(p.handle) == vx.VX_OK
    _, n_after, _, _ = vx.vx_table_info(p.handle, vx.VX_TABLE2)
    assert n_after == n2
    t2 = p.t2.cpu().numpy()
    return p, t2, work


CASES = [(1, 0, {}), (5, 3, {}), (11, 5, {}), (12, 6, {}), (14, 8, {}), (16, 9, {}), (18, 10, {}),
         (20, 11, {}), (22, 0, {}), (22, 1, dict(match_scope=1)), (18, 12, dict(partition_log2=8)),
         (17, 18, dict(scatter_mode=2)), (16, 22, dict(fuse_pair_hash=1)),
         (14, 8, dict(t2_placement=2)), (19, 13, dict(match_scope=1, partition_log2=7))]


@pytest.mark.parametrize("K,seed,kw", CASES)
def test_sort_table2_matches_oracle(vx, K, seed, kw):
    key = plot_key(seed)
    p, got, _ = sorted_plot(vx, K, key, kw)
    t1 = orc.table1(K, key)
    D = orc.default_distance(K)
    ref = orc.match_global(key, t1, D) if kw.get("match_scope") else orc.match(key, t1, D)
    assert np.array_equal(got, orc.sort_table2(ref))
    p.close()


@pytest.mark.parametrize("K,mult", [(4, 2), (10, 1), (10, 2), (12, 3), (16, 4), (21, 1), (21, 2)])
def test_sort_table2_levels_and_fills(vx, K, mult):
    # One partition of few records and of more than its digits' words like
    # (several pairs per record), one scatter level with a partial last tile,
    # 10 partition bits in one level and, from 2^21 records on, 11 in two.
    key = plot_key(60 + K)
    D = mult * orc.default_distance(K)
    p, got, _ = sorted_plot(vx, K, key, dict(match_scope=1, match_distance=D, t2_capacity=(mult + 1) << K))
    ref = orc.sort_table2(orc.match_global(key, orc.table1(K, key), D))
    assert K < 21 or (got.shape[0] >= 1 << 21) == (mult == 2)
    assert np.array_equal(got, ref)
    p.close()


def test_sort_table2_after_split_path_and_twice(vx):
    K, key = 20, plot_key(44)
    p, got, work = sorted_plot(vx, K, key, {}, split=True)
    ref = orc.sort_table2(orc.match(key, orc.table1(K, key), orc.default_distance(K)))
    assert np.array_equal(got, ref)
    # sorting the sorted table again changes nothing
    vx.vx_sort_table2(p.handle, work.data_ptr(), work.numel())
    assert vx.vx_sync(p.handle) == vx.VX_OK
    assert np.array_equal(p.t2.cpu().numpy(), ref)
    p.close()


def test_sort_table2_call_errors(vx):
    p = vx.Plot(14, plot_key(45))
    # not run / not synced yet
    with pytest.raises(vx.VxError) as ei:
        vx.vx_sort_table2_work_bytes(p.handle)
    assert ei.value.code == vx.VX_ENOTREADY
    p.run()
    p.sync()
    wb = vx.vx_sort_table2_work_bytes(p.handle)
    work = torch.empty(wb, dtype=torch.uint8, device="cuda")
    assert vx.lib().vx_sort_table2(p.handle, work.data_ptr(), wb - 256, None) == vx.VX_EINVAL
    assert vx.lib().vx_sort_table2(p.handle, work.data_ptr() + 8, wb - 256, None) == vx.VX_EINVAL
    p.close()


@pytest.mark.parametrize("placement", [0, 1], ids=["slots", "lookback"])
def test_sort_table2_of_plots_that_only_ran_in_a_batch(vx, placement):
    # look-back batches leave no results in the plots' pinned blocks: a handle
    # that never ran alone has none when its Table 2 is sorted
    mix = [(16, 70), (14, 71)]
    plots = [vx.Plot(K, plot_key(s), vx.make_opts(t2_placement=placement)) for K, s in mix]
    vx.vx_plot_batch([p.handle for p in plots])
    for (K, s), p in zip(mix, plots):
        n2 = p.sync()
        wb = vx.vx_sort_table2_work_bytes(p.handle)
        work = torch.empty(max(wb, 256), dtype=torch.uint8, device="cuda")
        vx.vx_sort_table2(p.handle, work.data_ptr(), wb)
        assert vx.vx_sync(p.handle) == vx.VX_OK
        assert vx.vx_table_info(p.handle, vx.VX_TABLE2)[1] == n2
        key = plot_key(s)
        ref = orc.sort_table2(orc.match(key, orc.table1(K, key), orc.default_distance(K)))
        assert np.array_equal(p.t2.cpu().numpy(), ref)
        p.close()


def test_sort_table2_after_another_plot_took_the_scratch(vx):
    # Plots A and B share Table 1 and scratch, each with its own Table 2: A's
    # sort, issued after B ran, orders A's records and reports A's counts.
    K = 18
    t1b, t2b, scb = vx.vx_plot_required_bytes(K)
    t1 = torch.empty(t1b, dtype=torch.uint8, device="cuda")
    sc = torch.empty(scb, dtype=torch.uint8, device="cuda")
    t2 = [torch.empty(t2b, dtype=torch.uint8, device="cuda") for _ in range(2)]
    keys = [plot_key(72), plot_key(73)]
    refs = [orc.match(k, orc.table1(K, k), orc.default_distance(K)) for k in keys]
    assert refs[0].shape[0] != refs[1].shape[0]
    hs = []
    for key, buf in zip(keys, t2):
        hs.append(vx.vx_plot_create(K, key))
        vx.vx_plot_bind(hs[-1], t1.data_ptr(), buf.data_ptr(), sc.data_ptr(), t2b // 16)
        vx.vx_plot_run(hs[-1])
        vx.vx_sync(hs[-1])
    for h, buf, ref in zip(hs, t2, refs):
        wb = vx.vx_sort_table2_work_bytes(h)
        work = torch.empty(wb, dtype=torch.uint8, device="cuda")
        vx.vx_sort_table2(h, work.data_ptr(), wb)
        assert vx.vx_sync(h) == vx.VX_OK
        n2 = vx.vx_table_info(h, vx.VX_TABLE2)[1]
        assert n2 == ref.shape[0]
        assert np.array_equal(buf[: 16 * n2].view(n2, 16).cpu().numpy(), orc.sort_table2(ref))
    for h in hs:
        vx.vx_plot_destroy(h)

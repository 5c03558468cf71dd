"""GPU parity of ss_embbag_fwd and ss_embbag_bwd_adagrad against the oracle."""
import numpy as np
import pytest
import torch

from oracle import shadowsync_oracle as O
from paper_2003_03477_b200 import binding as ss
from paper_2003_03477_b200 import synth
from parity import RTOL_F32, assert_close

pytestmark = pytest.mark.gpu


def _cuda(a, dt=None):
    t = torch.from_numpy(np.ascontiguousarray(a)).cuda()
    return t if dt is None else t.to(dt)


def _fwd(tables, idx, off, B, col0=None, want_bf16=False):
    T, N, D = tables.shape
    col0 = D if col0 is None else col0
    W = col0 + T * D
    out = torch.full((B, W), -7.0, device="cuda")
    outh = torch.zeros(B, W, dtype=torch.bfloat16, device="cuda") if want_bf16 else None
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    ss.ss_embbag_fwd(_cuda(tables), T, N, D, _cuda(idx), _cuda(off), B, out, W, outh, W, col0, st)
    torch.cuda.synchronize()
    return out.cpu().numpy(), (outh.float().cpu().numpy() if want_bf16 else None), int(st.item())


@pytest.mark.parametrize("D", [4, 8, 16, 64, 128, 256])
def test_fwd_parity_small(D):
    cfg = synth.scaled(synth.CONFIGS["tiny"], T=3, N=500, D=D, B=37, bottom=(13, 64, D), top=(4 * D, 64, 1))
    b = synth.make_batch(cfg, 0, 0)
    tables = synth.tables_dense(cfg)
    want = O.embbag_fwd(tables, b.indices, b.offsets, cfg.B)
    got, goth, st = _fwd(tables, b.indices, b.offsets, cfg.B, want_bf16=True)
    assert st == 0
    assert_close(got[:, D:], want.reshape(cfg.B, -1), RTOL_F32, "pooled")
    assert (got[:, :D] == -7.0).all()                     # columns before col0 are not touched
    assert np.array_equal(goth[:, D:], torch.from_numpy(got[:, D:]).to(torch.bfloat16).float().numpy())


def test_fwd_tiny_config_full():
    cfg = synth.CONFIGS["tiny"]
    b = synth.make_batch(cfg, 1, 3)
    tables = synth.tables_dense(cfg)
    want = O.embbag_fwd(tables, b.indices, b.offsets, cfg.B)
    got, _, st = _fwd(tables, b.indices, b.offsets, cfg.B)
    assert st == 0
    assert_close(got[:, cfg.D:], want.reshape(cfg.B, -1), RTOL_F32, "pooled")


def test_fwd_edge_cases_empty_bags_single_row_duplicates_and_bad_index():
    tables = np.random.default_rng(0).normal(size=(2, 7, 8)).astype(np.float32)
    # table 0: bag0 = [], bag1 = [3], bag2 = [5, 5, 5]; table 1: bag0 = [6, 0], bag1 = [], bag2 = [9 (bad), 1]
    idx = np.array([3, 5, 5, 5, 6, 0, 9, 1], np.int32)
    off = np.array([0, 0, 1, 4, 6, 6, 8], np.int32)
    got, _, st = _fwd(tables, idx, off, 3, col0=0)
    assert st == ss.SS_DEV_BAD_INDEX
    assert not got[0, :8].any() and np.array_equal(got[1, :8], tables[0, 3])
    assert_close(got[2, :8], 3.0 * tables[0, 5].astype(np.float64), RTOL_F32)
    assert_close(got[0, 8:], tables[1, 6].astype(np.float64) + tables[1, 0], RTOL_F32)
    assert not got[1, 8:].any() and np.array_equal(got[2, 8:], tables[1, 1])   # the bad lookup is skipped
    # all-ones table: pooled = bag length exactly
    ones = np.ones((2, 7, 8), np.float32)
    idx[6] = 2
    got, _, st = _fwd(ones, idx, off, 3, col0=0)
    assert st == 0 and np.array_equal(got[:, 0], [0, 1, 3]) and np.array_equal(got[:, 8], [2, 0, 2])


def test_fwd_malformed_offsets_give_empty_bags_and_a_status_bit():
    """Offsets that decrease, are negative or point beyond the end of the index list (offsets[T*B]) must not
    become reads outside the list: such a bag pools to zero and SS_DEV_BAD_OFFSET is raised; the well-formed
    bags of the same call are unaffected."""
    tables = np.random.default_rng(1).normal(size=(1, 7, 8)).astype(np.float32)
    idx = np.array([3, 5, 6, 1], np.int32)
    for off, bad_bags in ((np.array([0, 1, 1 << 30, 3, 4], np.int32), (1, 2)),     # far beyond the list
                          (np.array([0, 2, 1, 3, 4], np.int32), (1,)),              # decreasing
                          (np.array([0, -5, 2, 3, 4], np.int32), (0, 1))):          # negative
        got, _, st = _fwd(tables, idx, off, 4, col0=0)
        assert st & ss.SS_DEV_BAD_OFFSET, off
        for b in range(4):
            if b in bad_bags:
                assert not got[b].any(), (off, b)
            else:
                want = tables[0, idx[off[b]:off[b + 1]]].astype(np.float64).sum(axis=0)
                assert_close(got[b], want, RTOL_F32, f"bag {b}", floor=1.0)


def _bwd(cfg, batch, tables, state, gp, keep=True):
    T, N, D, B, L = cfg.T, cfg.N, cfg.D, cfg.B, batch.L
    dt, ds = _cuda(tables), _cuda(state.reshape(-1))
    ws = torch.empty(ss.ss_embbag_bwd_workspace_bytes(T, N, D, B, L), dtype=torch.uint8, device="cuda")
    uniq = torch.full((max(L, 1),), -1, dtype=torch.int32, device="cuda")
    seg = torch.full((L + 1,), -1, dtype=torch.int32, device="cuda")
    perm = torch.full((max(L, 1),), -1, dtype=torch.int32, device="cuda")
    nu = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    ss.ss_embbag_bwd_adagrad(dt, ds, T, N, D, _cuda(batch.indices), _cuda(batch.offsets), B, L, _cuda(gp), T * D, 0,
                             cfg.lr, cfg.eps, ws, uniq, seg, perm, nu, st)
    torch.cuda.synchronize()
    U = int(nu.item())
    return (dt.cpu().numpy(), ds.cpu().numpy().reshape(T, N), uniq.cpu().numpy()[:U], seg.cpu().numpy()[:U + 1],
            perm.cpu().numpy()[:L], int(st.item()))


def _check_bwd(cfg, step=0, seed=0):
    b = synth.make_batch(cfg, 0, step)
    tables = synth.tables_dense(cfg)
    rng = np.random.default_rng(seed)
    state = (rng.random((cfg.T, cfg.N)) * 1e-4).astype(np.float32)
    gp = (rng.normal(size=(cfg.B, cfg.T * cfg.D)) * 1e-3).astype(np.float32)
    t_o, s_o = tables.copy(), state.copy()
    uniq, seg, perm = O.embbag_bwd_adagrad(t_o, s_o, b.indices, b.offsets, cfg.B, gp, cfg.lr, cfg.eps)
    t_g, s_g, uniq_g, seg_g, perm_g, st = _bwd(cfg, b, tables, state, gp)
    assert st == 0
    # integer outputs are bit-exact
    assert np.array_equal(uniq_g, uniq) and np.array_equal(seg_g, seg) and np.array_equal(perm_g, perm)
    # the update is compared on the *change* of the touched rows and on the state
    assert_close(t_g - tables, t_o.astype(np.float64) - tables, 2e-5, "table update")
    assert_close(s_g, s_o, RTOL_F32, "row state")
    untouched = np.ones((cfg.T, cfg.N), bool)
    untouched[uniq // cfg.N, uniq % cfg.N] = False
    assert np.array_equal(t_g[untouched], tables[untouched])
    return len(uniq), b.L


@pytest.mark.parametrize("D", [4, 16, 64, 128])
def test_bwd_parity_small_uniform(D):
    cfg = synth.scaled(synth.CONFIGS["tiny"], T=3, N=300, D=D, B=64, bottom=(13, 64, D), top=(4 * D, 64, 1))
    U, L = _check_bwd(cfg)
    assert U < L            # 300 rows per table: duplicates, segments longer than one


def test_bwd_parity_skewed_long_segments_cross_windows_and_sort_tiles():
    # Zipf rows: the hottest row of each table has hundreds of lookups -> runs spanning many 16-wide windows;
    # about 5k lookups per table: the per-table shared-memory sort takes them (the tiled passes are covered by the
    # malformed-input cases, the no-scratch entry point and the full-size test of the large workload)
    cfg = synth.scaled(synth.CONFIGS["medium"], T=4, N=20_000, D=64, B=512, bottom=(13, 64, 64), top=(320, 64, 1))
    U, L = _check_bwd(cfg)
    assert L > 4 * 4096 and U < L // 2


def test_bwd_tiny_config_full():
    _check_bwd(synth.CONFIGS["tiny"], step=2)


def test_bwd_edge_cases():
    # one row hit by every bag; bags of length 1; an empty table slice; a bad index
    T, N, D, B = 3, 50, 8, 40
    cfg = synth.scaled(synth.CONFIGS["tiny"], T=T, N=N, D=D, B=B)
    idx0 = np.full(B, 7, np.int32)                               # table 0: every bag hits row 7
    idx2 = (np.arange(B) % N).astype(np.int32)                   # table 2: bags of one lookup
    idx = np.concatenate([idx0, idx2])
    off = np.concatenate([np.arange(B + 1), np.full(B, B), B + 1 + np.arange(B)]).astype(np.int32)  # table 1 empty
    batch = synth.Batch(idx, off, np.zeros((B, 13), np.float32), np.zeros(B, np.float32))
    tables = synth.tables_dense(cfg)
    state = np.zeros((T, N), np.float32)
    gp = np.random.default_rng(1).normal(size=(B, T * D)).astype(np.float32)
    t_o, s_o = tables.copy(), state.copy()
    uniq, seg, perm = O.embbag_bwd_adagrad(t_o, s_o, idx, off, B, gp, cfg.lr, cfg.eps)
    t_g, s_g, uniq_g, seg_g, perm_g, st = _bwd(cfg, batch, tables, state, gp)
    assert st == 0 and np.array_equal(uniq_g, uniq) and np.array_equal(seg_g, seg) and np.array_equal(perm_g, perm)
    assert uniq[0] == 7 and seg[1] == B
    assert_close(t_g - tables, t_o.astype(np.float64) - tables, 2e-5, "table update")
    assert_close(s_g, s_o, RTOL_F32, "row state")
    # a bad index is flagged and skipped; the remaining lookups give the oracle's result on the cleaned input
    idx_bad = idx.copy()
    idx_bad[3] = N + 5
    batch_bad = synth.Batch(idx_bad, off, batch.dense, batch.labels)
    t_g, s_g, uniq_g, seg_g, perm_g, st = _bwd(cfg, batch_bad, tables, state, gp)
    assert st == ss.SS_DEV_BAD_INDEX
    assert seg_g[-1] == len(idx) - 1 and uniq_g[0] == 7 and seg_g[1] == B - 1
    assert 3 not in perm_g[: seg_g[-1]]


def test_bwd_empty_input():
    cfg = synth.scaled(synth.CONFIGS["tiny"], T=2, N=10, D=8, B=4)
    batch = synth.Batch(np.zeros(0, np.int32), np.zeros(9, np.int32), np.zeros((4, 13), np.float32), np.zeros(4, np.float32))
    tables = synth.tables_dense(cfg)
    t_g, s_g, uniq_g, seg_g, perm_g, st = _bwd(cfg, batch, tables, np.zeros((2, 10), np.float32),
                                                np.ones((4, 16), np.float32))
    assert st == 0 and len(uniq_g) == 0 and list(seg_g) == [0] and np.array_equal(t_g, tables)


def test_device_table_fill_matches_host_generator():
    from paper_2003_03477_b200 import trainer
    cfg = synth.scaled(synth.CONFIGS["tiny"], T=3, N=1000, D=16)
    dev = trainer.device_tables(cfg).cpu().numpy()
    assert np.array_equal(dev, synth.tables_dense(cfg))


def test_sort_once_apply_twice_matches_two_oracle_updates():
    # the two-call form: the sort half fills the workspace, the apply half may be repeated on it
    cfg = synth.scaled(synth.CONFIGS["medium"], T=3, N=4000, D=64, B=256, bottom=(13, 64, 64), top=(256, 64, 1))
    b = synth.make_batch(cfg, 0, 1)
    tables = synth.tables_dense(cfg)
    state = np.zeros((cfg.T, cfg.N), np.float32)
    rng = np.random.default_rng(3)
    gp = (rng.normal(size=(cfg.B, cfg.T * cfg.D)) * 1e-3).astype(np.float32)
    t_o, s_o = tables.copy(), state.copy()
    for _ in range(3):
        uniq, seg, perm = O.embbag_bwd_adagrad(t_o, s_o, b.indices, b.offsets, cfg.B, gp, cfg.lr, cfg.eps)
    T, N, D, B, L = cfg.T, cfg.N, cfg.D, cfg.B, b.L
    dt, ds = _cuda(tables), _cuda(state.reshape(-1))
    ws = torch.empty(ss.ss_embbag_bwd_workspace_bytes(T, N, D, B, L), dtype=torch.uint8, device="cuda")
    nu = torch.zeros(1, dtype=torch.int32, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    perm_d = torch.empty(L, dtype=torch.int32, device="cuda")
    ss.ss_embbag_bwd_sort(T, N, D, _cuda(b.indices), _cuda(b.offsets), B, L, ws, None, None, perm_d, nu, st)
    dg = _cuda(gp)
    for _ in range(3):
        ss.ss_embbag_bwd_apply(dt, ds, T, N, D, B, L, dg, T * D, 0, cfg.lr, cfg.eps, ws, st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0 and int(nu.item()) == len(uniq) and np.array_equal(perm_d.cpu().numpy(), perm)
    assert_close(dt.cpu().numpy() - tables, t_o.astype(np.float64) - tables, 2e-5, "tables after three updates")
    assert_close(ds.cpu().numpy().reshape(T, N), s_o, RTOL_F32, "row state")


def test_apply_refuses_a_workspace_sorted_for_another_problem():
    # the apply half trusts the workspace only if the sort stamped it for the same T, N, L
    cfg = synth.scaled(synth.CONFIGS["medium"], T=3, N=4000, D=64, B=256, bottom=(13, 64, 64), top=(256, 64, 1))
    b1, b2 = synth.make_batch(cfg, 0, 1), synth.make_batch(cfg, 0, 2)
    assert b1.L != b2.L
    T, N, D, B = cfg.T, cfg.N, cfg.D, cfg.B
    Lmax = max(b1.L, b2.L)
    tables = synth.tables_dense(cfg)
    dt, ds = _cuda(tables), torch.zeros(T * N, device="cuda")
    ws = torch.zeros(ss.ss_embbag_bwd_workspace_bytes(T, N, D, B, Lmax), dtype=torch.uint8, device="cuda")
    nu = torch.zeros(1, dtype=torch.int32, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    dg = torch.ones(B, T * D, device="cuda")
    # never sorted: refused
    ss.ss_embbag_bwd_apply(dt, ds, T, N, D, B, b1.L, dg, T * D, 0, 0.1, 1e-8, ws, st)
    torch.cuda.synchronize()
    assert int(st.item()) == ss.SS_DEV_BAD_WORKSPACE and np.array_equal(dt.cpu().numpy(), tables)
    # sorted for batch 1, applied with batch 2's size: refused, tables untouched
    st.zero_()
    ss.ss_embbag_bwd_sort(T, N, D, _cuda(b1.indices), _cuda(b1.offsets), B, b1.L, ws, None, None, None, nu, st)
    ss.ss_embbag_bwd_apply(dt, ds, T, N, D, B, b2.L, dg, T * D, 0, 0.1, 1e-8, ws, st)
    torch.cuda.synchronize()
    assert int(st.item()) == ss.SS_DEV_BAD_WORKSPACE and np.array_equal(dt.cpu().numpy(), tables)
    # matching call goes through
    st.zero_()
    ss.ss_embbag_bwd_apply(dt, ds, T, N, D, B, b1.L, dg, T * D, 0, 0.1, 1e-8, ws, st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0 and not np.array_equal(dt.cpu().numpy(), tables)


def _run_lengths_batch(D, lengths, B, seed, spare=0):
    """Two tables whose rows are looked up `lengths` times each, cut into B bags at random places (some are empty)."""
    T, N = 2, len(lengths) + 3 + spare
    cfg = synth.scaled(synth.CONFIGS["tiny"], T=T, N=N, D=D, B=B, bottom=(13, 64, D), top=(3 * D, 64, 1))
    rng = np.random.default_rng(seed)
    idx, off = [], [0]
    for t in range(T):
        rows = np.repeat(np.arange(len(lengths), dtype=np.int32) + t, lengths)
        rng.shuffle(rows)
        cuts = np.sort(rng.integers(0, len(rows) + 1, B - 1))
        off += list(off[0] + len(idx) + np.append(cuts, len(rows)))
        idx += list(rows)
    return cfg, synth.Batch(np.array(idx, np.int32), np.array(off, np.int32), np.zeros((B, 13), np.float32),
                            np.zeros(B, np.float32))


# row widths on both sides of every lane mapping (4, 8, 16, 32 lanes' worth of float4, more than 256 floats), and row
# frequencies around the window (16 positions), the block's windows, and the longest span that is added beside the window (8)
@pytest.mark.parametrize("D", [4, 12, 16, 20, 32, 36, 64, 68, 128, 132, 200, 256, 260])
def test_bwd_runs_around_windows_blocks_and_spans(D):
    for seed, extra in ((1, []), (2, [1] * 37), (3, [16] * 33)):
        _check_runs(D, extra + RUN_LENGTHS, seed)


# the same with as many windows per SM as the fused kernel wants of rows of 129 to 256 floats, and as its forms for many windows
# want; rows that nobody looks up keep the lookups per row low enough for the fused kernel
@pytest.mark.parametrize("D,per_sm,spare", [(132, 16, True), (200, 16, True), (256, 16, True), (132, 29, True), (256, 29, True),
                                            (132, 16, False), (256, 29, False), (20, 121, False), (32, 121, False),
                                            (12, 33, False), (16, 33, False), (48, 17, False), (64, 17, False), (100, 17, False), (128, 17, False)])
def test_bwd_runs_with_many_windows(D, per_sm, spare):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    lengths = [5] + RUN_LENGTHS * (-(-per_sm * sms * 16 // (2 * sum(RUN_LENGTHS))) + 1)
    _check_runs(D, lengths, 4, sum(lengths) // 32 if spare else 0)


def _update_us(T, N, D, lookups, bag):
    """us of the update half for T tables of N rows, all about equally often looked up."""
    B = lookups // bag
    g = torch.Generator(device="cuda").manual_seed(1)
    off = torch.arange(0, T * B * bag + 1, bag, device="cuda").int()
    idx = torch.randint(0, N, (T * B * bag,), generator=g, device="cuda").int()
    tables, state = torch.zeros(T, N, D, device="cuda"), torch.ones(T * N, device="cuda")
    grad, st = torch.randn(B, T * D, generator=g, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(ss.ss_embbag_bwd_workspace_bytes(T, N, D, B, idx.numel()), dtype=torch.uint8, device="cuda")
    ss.ss_embbag_bwd_sort(T, N, D, idx, off, B, idx.numel(), ws, None, None, None, None, st)
    return _best_us(lambda: ss.ss_embbag_bwd_apply(tables, state, T, N, D, B, idx.numel(), grad, T * D, 0, 0.01, 1e-8, ws, st))


def _best_us(call):
    times = []
    for _ in range(20):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(10):
            call()
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b) * 100)
    return min(times)


# popular rows are summed, not updated lookup by lookup: what is left is reading the gradients.  Rows of 132 floats, 66 lookups of
# each row against one: 0.66 of the time where the fused kernel took both, 0.45 now
def test_bwd_of_popular_wide_rows_takes_the_time_of_their_gradients():
    assert _update_us(12, 300, 132, 20_000, 10) <= 0.55 * _update_us(12, 20_000, 132, 20_000, 10)


RUN_LENGTHS = [15, 1, 16, 16, 32, 17, 128, 1, 127, 2, 144, 7, 113, 1, 129, 3, 1, 1, 1, 260, 12, 33, 111, 1, 5, 600, 31, 96,
               97, 1, 14, 16, 48, 2, 1, 1, 1040, 30, 18, 112, 113]


def _check_runs(D, lengths, seed, spare=0):
    cfg, b = _run_lengths_batch(D, lengths, 61, seed, spare)
    rng = np.random.default_rng(seed)
    tables = (rng.normal(size=(cfg.T, cfg.N, D)) * 0.05).astype(np.float32)
    state = (rng.random((cfg.T, cfg.N)) * 1e-4).astype(np.float32)
    gp = (rng.normal(size=(cfg.B, cfg.T * D)) * 1e-3).astype(np.float32)
    t_o, s_o = tables.copy(), state.copy()
    uniq, seg, _ = O.embbag_bwd_adagrad(t_o, s_o, b.indices, b.offsets, cfg.B, gp, cfg.lr, cfg.eps)
    t_g, s_g, uniq_g, seg_g, _, st = _bwd(cfg, b, tables, state, gp)
    assert st == 0 and np.array_equal(uniq_g, uniq) and np.array_equal(seg_g, seg)
    # a row's sum has up to 1040 terms, added in two levels of at most 65 and 16: 81 * 2^-24 = 5e-6 of their size
    assert_close(t_g - tables, t_o.astype(np.float64) - tables, 3e-5, f"table update, {seed}")
    assert_close(s_g, s_o, 2e-5, f"row state, {seed}")


# bag lengths around the rounds of the gather, odd batches (the last block is not full)
@pytest.mark.parametrize("D", [4, 16, 20, 32, 64, 68, 128, 132, 200, 256, 260, 512])
def test_fwd_bags_around_the_rounds_of_the_gather(D):
    rng = np.random.default_rng(D)
    T, N, lens = 2, 97, [0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 11, 12, 13, 16, 17, 18, 19, 0, 24, 25, 40, 1, 0]
    B = len(lens)
    tables = rng.normal(size=(T, N, D)).astype(np.float32)
    off = np.concatenate([[0], np.cumsum(lens + lens)]).astype(np.int32)
    idx = rng.integers(0, N, off[-1]).astype(np.int32)
    want = O.embbag_fwd(tables, idx, off, B)
    got, goth, st = _fwd(tables, idx, off, B, col0=0, want_bf16=True)
    assert st == 0
    # up to 40 terms of size one added in float: 40 * 2^-24 = 2.4e-6 of the sum's scale, sqrt(40)
    assert_close(got, want.reshape(B, -1), RTOL_F32, "pooled", floor=1.0)
    assert np.array_equal(goth, torch.from_numpy(got).to(torch.bfloat16).float().numpy())


# a call with enough bags for the form whose blocks take stretches of consecutive bags (rows of 65 to 256 floats): stretches
# that end inside a table, an odd batch, empty bags, and batches smaller than a block's lane groups (many tables)
@pytest.mark.parametrize("D,T", [(64, 7), (68, 600), (100, 2), (128, 7), (132, 5), (200, 1200), (256, 3)])
def test_fwd_stretches_of_bags_match_the_sum_of_their_rows(D, T):
    lanes = 16 if D <= 128 else 32
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    B = sms * 2048 // lanes // T + 3
    g = torch.Generator(device="cuda").manual_seed(D)
    N = 61
    tables = torch.randn(T, N, D, generator=g, device="cuda")
    lens = torch.randint(0, 9, (T * B,), generator=g, device="cuda")
    off = torch.zeros(T * B + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=off[1:])
    idx = torch.randint(0, N, (int(off[-1]),), generator=g, device="cuda")
    table = torch.repeat_interleave(torch.arange(T * B, device="cuda") // B, lens)
    want = torch.nn.functional.embedding_bag(idx + table * N, tables.double().view(T * N, D), off, mode="sum", include_last_offset=True)
    out = torch.full((B, T * D + 4), -7.0, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    outh = torch.full((B, T * D + 12), -7.0, dtype=torch.bfloat16, device="cuda")
    i32, o32 = idx.int(), off.int()
    ss.ss_embbag_fwd(tables, T, N, D, i32, o32, B, out, T * D + 4, outh, T * D + 12, 4, st)
    assert int(st.item()) == 0 and bool((out[:, :4] == -7.0).all()) and bool((outh[:, :4] == -7.0).all())
    assert torch.equal(outh[:, 4:4 + T * D], out[:, 4:].bfloat16()) and bool((outh[:, 4 + T * D:] == -7.0).all())
    got = out[:, 4:].view(B, T, D).transpose(0, 1).reshape(T * B, D).double()
    # up to 8 terms of size one: 8 * 2^-24 of the sum of their magnitudes, at most 8 * 5
    assert float((got - want).abs().max()) <= 2e-5
    # an index outside a table and a decreasing offset: skipped, and said so; the other bags are as before
    bags = torch.nonzero(lens > 1).flatten()
    bad_bag, cut = int(bags[0]), int(bags[len(bags) // 2])
    i32[int(off[bad_bag])] = N
    o32[cut + 1] = o32[cut] - 1
    ss.ss_embbag_fwd(tables, T, N, D, i32, o32, B, out, T * D + 4, None, 0, 4, st)
    assert int(st.item()) == ss.SS_DEV_BAD_INDEX | ss.SS_DEV_BAD_OFFSET
    again = out[:, 4:].view(B, T, D).transpose(0, 1).reshape(T * B, D).double()
    rest = want[bad_bag] - tables[bad_bag // B, idx[off[bad_bag]]].double()
    assert float((again[bad_bag] - rest).abs().max()) <= 2e-5 and not bool(again[cut].any())
    same = torch.ones(T * B, dtype=torch.bool, device="cuda")
    same[[bad_bag, cut, cut + 1]] = False
    assert torch.equal(again[same], got[same])


def _csr_batch(lens, N, D, T, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    off = torch.zeros(lens.numel() + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=off[1:])
    idx = torch.randint(0, N, (int(off[-1]),), generator=g, device="cuda")
    return torch.randn(T, N, D, generator=g, device="cuda"), idx, off


def _uneven(kind, T, B, g):
    """Bag lengths of T tables that differ in them."""
    t = torch.arange(T, device="cuda").view(T, 1).expand(T, B)
    r = torch.rand(T, B, generator=g, device="cuda")
    lens = {"one_long": torch.where(t == T // 2, 40, 2), "first_long": torch.where(t == 0, 40, 1), "last_long": torch.where(t == T - 1, 40, 0),
            "halves": torch.where(t < T // 2, 1, 9), "by_table": t % 23, "one_lookup": torch.ones_like(t), "one_bag": (r == r.max()) * 60_000,
            "few_long_bags": torch.where(r < 0.01, 100, (r * 3).long()), "empty": torch.zeros_like(t)}[kind]
    return lens.reshape(-1).long()


# the same form where tables differ in bag length: its stretches are cut by work, short bags are summed two at a time
@pytest.mark.parametrize("kind", ["one_long", "first_long", "last_long", "halves", "by_table", "one_lookup", "one_bag", "few_long_bags", "empty"])
@pytest.mark.parametrize("D,T", [(128, 7), (100, 300), (256, 3)])
def test_fwd_stretches_of_uneven_tables(D, T, kind):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    B = sms * 2048 // (16 if D <= 128 else 32) // T + 3
    N = 61
    lens = _uneven(kind, T, B, torch.Generator(device="cuda").manual_seed(D))
    tables, idx, off = _csr_batch(lens, N, D, T, D)
    table = torch.repeat_interleave(torch.arange(T * B, device="cuda") // B, lens)
    want = torch.nn.functional.embedding_bag(idx + table * N, tables.double().view(T * N, D), off, mode="sum", include_last_offset=True)
    i32, o32, st = torch.cat([idx, idx[:1], torch.zeros(1, dtype=idx.dtype, device="cuda")])[:max(idx.numel(), 1)].int(), off.int(), torch.zeros(1, dtype=torch.int32, device="cuda")
    out = torch.full((B, T * D), -7.0, device="cuda")
    ss.ss_embbag_fwd(tables, T, N, D, i32, o32, B, out, T * D, None, 0, 0, st)
    got = out.view(B, T, D).transpose(0, 1).reshape(T * B, D).double()
    assert int(st.item()) == 0
    # n terms of size up to 5 added in float: n * 2^-24 of 5 n at most; sums of n random terms stay far below that bound
    n = lens.max().clamp(min=1).double()
    assert float((got - want).abs().max()) <= float(n * 2.0 ** -24 * 5 * n.sqrt() * 4)
    # offsets that ascend nowhere near everywhere: every bag is written all the same, the sound ones with their sums
    g = torch.Generator(device="cuda").manual_seed(1)
    at = torch.randint(0, T * B, (max(T * B // 3, 1),), generator=g, device="cuda")
    o32[at] = torch.randint(-2 ** 31, 2 ** 31 - 1, at.shape, generator=g, device="cuda").int()
    out.fill_(-7.0)
    st.zero_()
    ss.ss_embbag_fwd(tables, T, N, D, i32, o32, B, out, T * D, None, 0, 0, st)
    again = out.view(B, T, D).transpose(0, 1).reshape(T * B, D).double()
    lo, hi, L = o32[:-1].long(), o32[1:].long(), int(off[-1])
    same = (lo == off[:-1]) & (hi == off[1:])
    empty = (lo < 0) | (hi < lo) | (hi > L)
    assert int(st.item()) & ss.SS_DEV_BAD_OFFSET and torch.equal(again[same], got[same]) and not bool(again[empty].any())


# the lookup's time follows its lookups, not which table they are in: an even batch and one with a table 20 times as long as the
# others take about the same for the same number of lookups (with blocks that take equal numbers of bags: 4.5 times)
def test_fwd_of_one_long_table_is_as_fast_as_of_even_ones():
    T, B, D, N = 26, 4096, 128, 100_000
    even, uneven = torch.full((T, B), 3, device="cuda"), torch.full((T, B), 2, device="cuda")
    even[:12] = 4
    uneven[T // 3] = 40
    us = []
    for lens in (even, uneven):
        tables, idx, off = _csr_batch(lens.reshape(-1), N, D, T, 5)
        i32, o32, st = idx.int(), off.int(), torch.zeros(1, dtype=torch.int32, device="cuda")
        out = torch.empty(B, T * D, dtype=torch.bfloat16, device="cuda")
        us.append(_best_us(lambda: ss.ss_embbag_fwd(tables, T, N, D, i32, o32, B, None, 0, out, T * D, 0, st)))
    assert us[1] <= 2 * us[0], us

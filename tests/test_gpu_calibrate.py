"""The calibration kernel at the sizes where its passes change: rows of a few
tokens, rows around a vector, a warp and a block, rows kept on chip and longer
ones, one and several CTAs per cluster, both block sizes; scores with few
distinct values (the exact refinement of the rank bins and of the top-B, with
ties across CTAs); every pooling width.

The selection is checked exactly: all groups get the same score row and every
token belongs to the current frame, so beta = D = 1 and s_bar is the row
itself in fp32 (means of 1, 4 or 8 equal numbers), and the kept set must be the
B largest with ties to the lower index.  MI is held to 1e-5 relative plus 1e-6
absolute: each of its at most 512 terms, of order 1 / N to 1, is rounded to
fp32."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import starkv_oracle as O
from paper_2606_01790_gb300 import starkv as sk
from paper_2606_01790_gb300 import synthetic as syn

import harness as H

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

R = C = 16


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def _row(lp, levels, seed):
    """lp positive scores: lognormal, or quantised to `levels` values."""
    rng = np.random.default_rng([lp, levels, seed])
    s = rng.lognormal(0.0, 0.4, lp)
    if levels:
        s = np.ceil(s / s.max() * levels) / levels
    return s.astype(np.float32)


def _seq(row, G, budget, slot, per_head, seed, w=8, side=R):
    lp = row.size
    rng = np.random.default_rng([lp, seed, 7])
    meta = np.zeros(lp + w, np.uint32)
    r, c = rng.integers(0, side, lp), rng.integers(0, side, lp)
    meta[:lp] = sk.pack_meta(np.ones(lp), np.zeros(lp), r, c)
    P = G if per_head else 1
    seq = sk.Seq(meta=sk.meta_tensor(meta).cuda(), L=lp + w, cur_frame=0, budget=budget, slot=slot,
                 S=torch.from_numpy(np.repeat(row[None], G, 0)[None]).cuda().contiguous(),
                 idx=torch.full((1, P, budget), -1, dtype=torch.int32, device="cuda"),
                 score=torch.zeros(1, P, lp, device="cuda"),
                 stats=torch.zeros(1, sk.stats_stride(G), device="cuda"))
    return seq, (r, c)


def _check(seq, cells, row, G, per_head, side=R, K=8, M=8):
    B = seq.budget
    order = np.lexsort((np.arange(row.size), -row.astype(np.float64)))
    want = np.sort(order[:B])
    for p in range(G if per_head else 1):
        np.testing.assert_array_equal(seq.idx[0, p].cpu().numpy(), want)
    stats = seq.stats[0].double().cpu().numpy()
    bins = O.rank_bins(row.astype(np.float64), K)
    mi = O.mutual_information(bins, O.spatial_cells(cells[0], cells[1], side, side, M), K, M * M)
    np.testing.assert_allclose(stats[8:8 + G], mi, rtol=1e-5, atol=1e-6 * K * M * M / 512)
    _, temp = O.entropy_temperature(row.astype(np.float64), 0.95, 1.05, 1e-12)
    got = seq.score[0].double().cpu().numpy()
    np.testing.assert_allclose(got, np.repeat((row.astype(np.float64) ** (1 / temp))[None], got.shape[0], 0), rtol=1e-5)


def _config(G, slots, per_head):
    return sk.Config(n_layers=1, n_heads=G, n_kv_heads=G, window=8, grid_rows=R, grid_cols=C, max_seqs=slots,
                     n_warmup=0, n_ramp=0, select_mode=sk.SELECT_PER_HEAD if per_head else sk.SELECT_GLOBAL)


SIZES = [1, 2, 3, 4, 5, 31, 32, 33, 127, 129, 513, 1027, 4097, 14000, 50001, 56097]


@pytest.mark.parametrize("levels", [0, 1, 3, 40], ids=["distinct", "equal", "3levels", "40levels"])
@pytest.mark.parametrize("G,per_head", [(1, False), (4, False), (4, True), (32, False)],
                         ids=["G1", "G4", "G4_per_head", "G32"])
def test_selection_is_exact_on_given_scores(G, per_head, levels):
    st = sk.init_state(_config(G, 1, per_head))
    for lp in SIZES:
        row = _row(lp, levels, G)
        for B in sorted({1, lp // 5, lp - 1, lp} - {0}):
            sk.reset_seq(st, 0)
            seq, cells = _seq(row, G, B, 0, per_head, G)
            sk.select(st, 0, [seq], sk.workspace(st, [seq]))
            torch.cuda.synchronize()
            sk.check_device_error(st)
            _check(seq, cells, row, G, per_head)


@pytest.mark.parametrize("levels", [0, 3], ids=["distinct", "3levels"])
def test_a_batch_with_more_ctas_than_sms(levels):
    """32 ragged rows of 8 groups (256 CTAs): the two-per-SM variant, rows on
    chip and, past its smaller capacity, read again from S."""
    G, n = 8, 32
    st = sk.init_state(_config(G, n, False))
    sizes = (SIZES + [7, 64, 255, 2000, 6001, 9999, 20011, 30002] * 2)[:n]
    rows = [_row(lp, levels, i) for i, lp in enumerate(sizes)]
    made = [_seq(row, G, max(1, row.size // 4), i, False, i) for i, row in enumerate(rows)]
    seqs = [m[0] for m in made]
    sk.select(st, 0, seqs, sk.workspace(st, seqs))
    torch.cuda.synchronize()
    sk.check_device_error(st)
    for (seq, cells), row in zip(made, rows):
        _check(seq, cells, row, G, False)


def _crowded_row(lp, n, equal, seed):
    """lp scores spread over four octaves, n of them eight units of the last place
    apart (all in one or two buckets of the first histogram), `equal` of these the same."""
    rng = np.random.default_rng([lp, n, equal, seed])
    s = np.exp2(rng.uniform(-4.0, 0.0, lp)).astype(np.float32)
    crowd = np.float32(0.3).view(np.uint32) + 8 * np.arange(n, dtype=np.uint32)
    crowd[n // 4:n // 4 + equal] = crowd[n // 4]
    s[rng.permutation(lp)[:n]] = crowd.view(np.float32)
    return s


@pytest.mark.parametrize("equal", [0, 600, 3000], ids=["distinct", "600equal", "3000equal"])
@pytest.mark.parametrize("lp", [5000, 14000, 56097])
@pytest.mark.parametrize("G,per_head", [(1, False), (4, False), (4, True), (32, False)],
                         ids=["G1", "G4", "G4_per_head", "G32"])
def test_a_crowded_bucket_is_split_again(G, per_head, lp, equal):
    """4000 scores in a bucket: its own key range gets a histogram, which is searched
    for the B-th token; with many equal ones among them a second one, down to one key."""
    st = sk.init_state(_config(G, 1, per_head))
    row = _crowded_row(lp, 4000, equal, G)
    above = int((row > np.float32(0.31)).sum())   # (the crowd lies between 0.3 and 0.301)
    for B in (above + 1, above + 700, above + 2000, above + 3999):
        sk.reset_seq(st, 0)
        seq, cells = _seq(row, G, B, 0, per_head, G)
        sk.select(st, 0, [seq], sk.workspace(st, [seq]))
        torch.cuda.synchronize()
        sk.check_device_error(st)
        _check(seq, cells, row, G, per_head)


def test_no_room_for_rows_on_chip():
    """The largest patch grid and joint histogram with more CTAs than SMs: no token
    of a row fits on chip, so that every pass reads S again and the fused scores
    wait in their output row.  (MI: up to 4096 terms, hence 8 times the absolute
    tolerance of the 512-cell histogram.)"""
    G, n, side, K, M = 8, 32, 128, 16, 16
    st = sk.init_state(dataclasses.replace(_config(G, n, False), grid_rows=side, grid_cols=side, mi_bins=K, mi_grid=M))
    sizes = (SIZES + [7, 64, 255, 2000, 6001, 9999, 20011, 30002] * 2)[:n]
    rows = [_row(lp, 0 if i % 2 else 40, i) for i, lp in enumerate(sizes)]
    made = [_seq(row, G, max(1, row.size // 4), i, False, i, side=side) for i, row in enumerate(rows)]
    seqs = [m[0] for m in made]
    sk.select(st, 0, seqs, sk.workspace(st, seqs))
    torch.cuda.synchronize()
    sk.check_device_error(st)
    for (seq, cells), row in zip(made, rows):
        _check(seq, cells, row, G, False, side, K, M)


@pytest.mark.parametrize("pool", [1, 3, 7, 9, 11, 31])
def test_pooling_widths(pool):
    """Windows inside the neighbouring vectors (up to 9 taps) and wider ones."""
    wl = dataclasses.replace(syn.WORKLOADS["tiny"], n_text=67)   # L_p = 571: a ragged last vector
    si = syn.make_sequence(wl)
    h = H.hyper(n_warmup=0, n_ramp=0, pool_kernel=pool)
    p = H.oracle_params(h)
    st = sk.init_state(H.gpu_config(wl, h))
    ds = H.device_seq(si, wl)
    sk.step(st, [ds.seq], sk.workspace(st, [ds.seq]))
    torch.cuda.synchronize()
    sk.check_device_error(st)
    ref = H.oracle_layer(si, 0, wl, O.LayerState.fresh(wl.n_kv_heads, wl.grid_rows, wl.grid_cols), p)
    np.testing.assert_allclose(ds.seq.S[0].double().cpu().numpy(), ref["S"], rtol=1e-4)
    sc = H.check_scores(ds.seq.score[0].double().cpu().numpy(), ref, ref["S"], si, 0, wl, p)
    assert sc["ok"], sc
    ix = H.check_index_set(ds.seq.idx[0].cpu().numpy(), ref, si.budget)
    assert ix["ok"], ix

"""GPU parity: the CUDA path, called through the C ABI, against the CPU oracle on the same seeded inputs.

Gates (from the benchmark spec): block lists bit-exact except pairs whose energy lies within 1e-3 relative
of the threshold (counted and excluded); attention given the same lists within 2e-2 max-abs (BF16 inputs)
or 6e-2 (FP8 inputs); LSE within 1e-3 relative.
"""
import os

import numpy as np
import pytest
import torch

from oracle import fp2_oracle as O
from paper_2608_19758_b200 import binding, inputs

pytestmark = pytest.mark.gpu

TOL_O = {"bf16": 2e-2, "fp8": 6e-2}
TOL_LSE_REL = 1e-3
NEAR_BAND = 1e-3


NEAR_SEEN = {}      # test id -> (excluded near-threshold mismatches, candidate pairs compared)


def make(spec, edit_case=None, **over):
    case = inputs.make_case(spec)
    if edit_case is not None:
        edit_case(case)   # e.g. other per-head scales: still a valid input, the oracle sees the same arrays
    dc = binding.DeviceCase(case, **over)
    dc.poison = True    # every stage call first overwrites what it is about to fill (lists -1, outputs NaN)
    prm = dict(case.params())
    prm.update(over)
    wl = O.Workload(O.Params.from_dict(prm), **inputs.oracle_args(case))
    return case, dc, wl


def check_lists(dc, wl, seg_ids=None, label=None):
    """Block lists of the GPU against the oracle's: bit-exact except for pairs whose energy lies within 1e-3
    relative of the threshold.  Those are counted, reported (printed, and kept in NEAR_SEEN) and excluded; their
    number is itself bounded: at most 1e-3 of the candidate pairs compared (plus one, for tiny cases).
    Returns (selected, excluded_near_threshold)."""
    off = dc.seg_offset.cpu().numpy()
    cnt = dc.seg_count.cpu().numpy()
    idx = dc.blk_idx.cpu().numpy()
    sel = O.oracle_select(wl, seg_ids)
    near = tot = cand = 0
    for seg, (oi, E, margin) in sel.items():
        assert 0 <= cnt[seg] <= len(E), f"segment {seg}: count {cnt[seg]}"
        g = idx[off[seg]:off[seg] + cnt[seg]]
        assert np.all(np.diff(g) > 0), f"segment {seg}: list not ascending"
        cand += len(E)
        tot += len(g)
        if len(g) == len(oi) and np.array_equal(g, oi):
            continue
        diff = np.setxor1d(g, oi)
        assert diff.min() >= 0 and diff.max() < len(E), f"segment {seg}: entry outside the candidates"
        bad = diff[margin[diff] > NEAR_BAND]
        assert bad.size == 0, f"segment {seg} block {bad[0]}: margin {margin[bad[0]]:.3e} outside the band"
        near += diff.size
    assert near <= 1 + 1e-3 * cand, f"{near} near-threshold exclusions among {cand} candidate pairs"
    name = label or os.environ.get("PYTEST_CURRENT_TEST", "?").split(" ")[0]
    NEAR_SEEN[name] = (near, cand)
    print(f"[lists] {name}: {near} near-threshold pairs excluded of {cand} candidate pairs compared, {tot} selected")
    return tot, near


def check_attention(dc, wl, lists, seg_ids=None, dense=False, dtype="bf16"):
    att = O.oracle_attend(wl, lists, seg_ids, dense=dense)
    tq = dc.case.total_q
    Oo, Lo = O.scatter_output(wl, att, tq)
    go = dc.out.float().cpu().numpy().astype(np.float64)
    gl = dc.lse.cpu().numpy().astype(np.float64)
    mask = ~np.isnan(Lo)
    assert mask.any()
    assert np.isfinite(go[mask.T]).all()
    err_o = np.abs(go - Oo)[mask.T].max()
    err_l = (np.abs(gl - Lo)[mask] / np.maximum(np.abs(Lo[mask]), 1.0)).max()
    assert err_o <= TOL_O[dtype], f"max-abs output error {err_o:.4f}"
    assert err_l <= TOL_LSE_REL, f"relative LSE error {err_l:.2e}"
    return err_o, err_l


def full_pipeline(spec, dense=True, edit_case=None, **over):
    case, dc, wl = make(spec, edit_case=edit_case, **over)
    dc.select()
    dc.status()
    check_lists(dc, wl)
    lists = dc.lists_host()
    dc.sparse()
    dc.status()
    check_attention(dc, wl, lists, dtype=spec.dtype)
    if dense:
        dc.dense()
        dc.status()
        check_attention(dc, wl, None, dense=True, dtype=spec.dtype)
    return case, dc, wl


# ------------------------------------------------------------------------------------------------------
# the named workloads
# ------------------------------------------------------------------------------------------------------

def test_config1_full():
    case, dc, wl = full_pipeline(inputs.config_spec(1))
    assert int(dc.seg_count.sum()) >= 364


def test_config2_full_lists_and_sparse_attention():
    spec = inputs.config_spec(2)
    case, dc, wl = make(spec)
    dc.select(); dc.status()
    tot, near = check_lists(dc, wl)
    pairs = dc.plan.idx_capacity
    assert pairs == 8 * 131584
    assert 0.04 < tot / pairs < 0.12
    lists = dc.lists_host()
    dc.sparse(); dc.status()
    check_attention(dc, wl, lists)
    # dense: sampled segments (first, last and random tiles of several heads)
    rng = np.random.default_rng(2)
    nt = 1024
    ids = sorted({h * nt + t for h in (0, 3, 7) for t in [0, 1, nt - 1] + rng.integers(0, nt, 3).tolist()})
    dc.dense(); dc.status()
    check_attention(dc, wl, None, ids, dense=True)


@pytest.mark.parametrize("alpha", [0.1, 1e-3])
def test_config3_relative_at_16k(alpha):
    spec = inputs.config_spec(3, scale_down=8)
    spec.alpha = alpha
    full_pipeline(spec, dense=(alpha == 0.1))


def test_config5_relative_batch_with_prefixes():
    spec = inputs.config_spec(5, scale_down=8)
    case, dc, wl = full_pipeline(spec)
    assert len(spec.seqs) == 16 and any(pre > 0 for _, pre in spec.seqs)


def _sampled_segments(wl, heads, tiles_per_head, seed):
    """First, last and random tiles of the given KV heads of sequence 0 (full-size workloads)."""
    rng = np.random.default_rng(seed)
    by_head = {}
    for s in wl.segs:
        if s.b == 0:
            by_head.setdefault(s.h, []).append(s.seg)
    ids = set()
    for h in heads:
        segs = by_head[h]
        n = len(segs)
        pick = {0, 1, n // 2, n - 2, n - 1} | set(rng.integers(0, n, tiles_per_head).tolist())
        ids |= {segs[i] for i in pick}
    return sorted(ids)


def _keep_widened_queries(wl):
    """The oracle widens all of q to fp64 on every call (4.3 GB at 131072 tokens x 32 heads); a test that calls it
    many times on one workload keeps the widened copy instead.  Same values, the oracle itself is untouched."""
    orig, kept = wl.q_seq, {}

    def q_seq(b):
        if b not in kept:
            kept[b] = orig(b)
        return kept[b]
    wl.q_seq = q_seq


def _set_alpha(dc, wl, alpha):
    """A new plan with another threshold on the same device tensors; the oracle reads alpha from its parameters."""
    prm = dict(dc.prm)
    prm["alpha"] = float(alpha)
    dc.plan.close()
    dc.plan = binding.Plan(prm, dc.case.cu_seqlens_q.tolist(), dc.case.seqlens_k.tolist())
    dc.prm = prm
    wl.p.alpha = float(alpha)


# thresholds that put the measured block sparsity of the 131072-token workloads near 50 / 75 / 90 / 95 / 98 %
# (bench.py finds its own by bisection; these are fixed so that the test does not depend on a search)
SWEEP_ALPHAS = {"bf16": [(0.50, 1.5e-5), (0.75, 1.8e-4), (0.90, 1.3e-3), (0.95, 4.6e-3), (0.98, 3.4e-2)],
                "fp8": [(0.50, 1.7e-5), (0.75, 1.9e-4), (0.90, 1.7e-3), (0.95, 6.3e-3), (0.98, 4.5e-2)]}


def _full_size_sweep(config, heads, seed):
    """One 131072-token workload in the launch configuration bench.py times.  At the headline threshold (95 %
    sparsity) the block lists of EVERY segment are compared with the oracle's; at every sweep point the lists and
    the attention output of sampled segments are; the dense path is compared on sampled segments."""
    spec = inputs.config_spec(config)
    dt = spec.dtype
    case, dc, wl = make(spec)
    _keep_widened_queries(wl)
    npairs = dc.plan.idx_capacity
    ids = _sampled_segments(wl, heads=heads, tiles_per_head=3, seed=seed)
    for target, alpha in SWEEP_ALPHAS[dt]:
        _set_alpha(dc, wl, alpha)
        dc.select(); dc.status()
        cnt = dc.seg_count.cpu().numpy()
        off = dc.seg_offset.cpu().numpy()
        idx = dc.blk_idx.cpu().numpy()
        assert off[-1] == npairs
        sparsity = 1.0 - cnt.sum() / npairs
        assert abs(sparsity - target) < 0.03, (target, sparsity)
        # any-size properties: counts within the candidates, diagonal band present, ascending
        for s in wl.segs[:: 97]:
            l = idx[off[s.seg]: off[s.seg] + cnt[s.seg]]
            assert 1 <= len(l) <= s.J_hi + 1 and np.all(np.diff(l) > 0) and l[-1] == s.J_hi
            assert set(range(s.J_lo, s.J_hi + 1)) <= set(l.tolist())
        if target == 0.95:
            check_lists(dc, wl, None, label=f"config {config} at 131072 tokens, alpha {alpha}: all segments")
        else:
            check_lists(dc, wl, ids, label=f"config {config} at 131072 tokens, alpha {alpha}: {len(ids)} segments")
        lists = {i: idx[off[i]: off[i] + cnt[i]].copy() for i in ids}
        dc.sparse(); dc.status()
        # the denser the lists, the fewer segments the oracle is asked for (one segment at 50 % is 2 GFLOP in fp64)
        att_ids = ids if target >= 0.9 else ids[:: 2]
        check_attention(dc, wl, lists, att_ids, dtype=dt)
        assert torch.isfinite(dc.out.float()).all() and torch.isfinite(dc.lse).all()
    dc.dense(); dc.status()
    check_attention(dc, wl, None, ids[:3] + ids[-2:], dense=True, dtype=dt)
    assert torch.isfinite(dc.out.float()).all()
    return dc, wl


def test_config3_full_size_all_lists_and_sweep_points():
    """BF16, 131072 tokens, Hq=32 / Hkv=8: 32768 segments, 16.8 M candidate pairs."""
    dc, wl = _full_size_sweep(3, heads=(0, 5), seed=3)
    assert dc.plan.idx_capacity == 8 * 2099200 and len(wl.segs) == 32768


def test_config5_full_size_sampled():
    """The continuous batch at full size (16 sequences, ~256K KV tokens, 16-token pages, prefixes)."""
    spec = inputs.config_spec(5)
    case, dc, wl = make(spec)
    dc.select(); dc.status()
    rng = np.random.default_rng(5)
    ids = sorted(set(rng.integers(0, len(wl.segs), 24).tolist()) | {0, len(wl.segs) - 1})
    check_lists(dc, wl, ids)
    lists_all = dc.lists_host()
    dc.sparse(); dc.status()
    check_attention(dc, wl, {i: lists_all[i] for i in ids}, ids)
    assert torch.isfinite(dc.out.float()).all()


# ------------------------------------------------------------------------------------------------------
# FP8 e4m3 inputs with per-head scales (Eq. 15); oracle on the de-quantised values
# ------------------------------------------------------------------------------------------------------

@pytest.mark.parametrize("g,hkv,p,seqs", [
    (7, 2, 64, [(2300, 0)]),
    (4, 2, 16, [(1500, 300), (700, 0), (129, 128)]),
    (1, 2, 32, [(900, 100)]),
])
def test_fp8_small(g, hkv, p, seqs):
    spec = inputs.small_spec(seqs=seqs, num_q_heads=g * hkv, num_kv_heads=hkv, page_size=p, dtype="fp8",
                             config_id=40 + g)
    spec.alpha = 0.2
    full_pipeline(spec)


def test_fp8_without_sink_and_heavy_pruning():
    spec = inputs.small_spec(seqs=[(4096, 0)], num_q_heads=8, num_kv_heads=2, page_size=64, dtype="fp8",
                             config_id=48, sink=False, sink_tokens=0, window_tokens=128)
    spec.alpha = 0.5
    case, dc, wl = full_pipeline(spec, dense=False)
    assert int(dc.seg_count.sum()) < dc.plan.idx_capacity / 2


@pytest.mark.parametrize("g,hkv,seqs", [
    (4, 2, [(1500, 300), (700, 0)]),
    (7, 1, [(1000, 0), (300, 100)]),
])
def test_fp8_query_scales_far_apart_within_a_group(g, hkv, seqs):
    """The heads of a group with query scales up to 30x apart (Eq. 15 gives every head its own): the scorer's
    reference maximum is then the exact one instead of the bound it uses for scales within a factor of two, and a
    packed tile's rows carry very different logit ranges through both kernels."""
    spec = inputs.small_spec(seqs=seqs, num_q_heads=g * hkv, num_kv_heads=hkv, page_size=16, dtype="fp8",
                             config_id=60 + g)
    spec.alpha = 0.1

    def spread(case):
        case.q_scale[1::2] *= 6.0
        case.q_scale[2::3] *= 0.2

    full_pipeline(spec, edit_case=spread)


@pytest.mark.parametrize("g", [1, 2, 3, 5, 7, 8, 9, 10, 16])
def test_fp8_row_multipliers_and_tiles_of_pairs(g):
    """FP8 scorer: row multipliers in registers (group sizes that divide 8, and 3, 5, 7, 10) or in shared memory (9, 16), with scales
    of their own for every head; query tiles widened one unit ahead, in pairs and singly, ragged last tiles.  There are five
    units for every CTA, so that both query buffers, both phases of their barriers and all four descriptors come round."""
    hkv, sms = 8, torch.cuda.get_device_properties(0).multi_processor_count
    lq = 10 * sms // hkv * 128 // g + 37
    while lq * g % 128 == 0 or -(-lq * g // 128) % 2 == 0:
        lq += 1                                          # a ragged last tile, one tile without a partner
    seqs = [(lq + 200, 200), (61, 0), (1300, 1290)]
    spec = inputs.small_spec(seqs=seqs, num_q_heads=g * hkv, num_kv_heads=hkv, page_size=16, dtype="fp8", config_id=240 + g)
    spec.alpha = 0.3

    def spread(case):
        case.q_scale[:] *= torch.linspace(0.5, 2.0, g * hkv)

    case, dc, wl = make(spec, edit_case=spread)
    tiles = [-(-(n - pre) * g // 128) for n, pre in seqs]
    assert dc.plan.num_segments == hkv * sum(tiles) > sms                     # so tiles are paired (all lists are short)
    assert hkv * sum(-(-t // 2) for t in tiles) >= 5 * sms
    dc.select()
    dc.status()
    check_lists(dc, wl)


def test_config4_relative_at_16k():
    spec = inputs.config_spec(4, scale_down=8)
    full_pipeline(spec)


def test_config4_full_size_all_lists_and_sweep_points():
    """FP8, 131072 tokens, Hq=28 / Hkv=4 (g = 7: tiles straddle positions): 28672 segments."""
    dc, wl = _full_size_sweep(4, heads=(1, 3), seed=4)
    assert len(wl.segs) == 28672


def test_config5_fp8_relative():
    spec = inputs.config_spec(5, dtype="fp8", scale_down=8)
    full_pipeline(spec)


# ------------------------------------------------------------------------------------------------------
# edge cases
# ------------------------------------------------------------------------------------------------------

@pytest.mark.parametrize("p", [8, 16, 32, 64, 128])
def test_page_sizes(p):
    spec = inputs.small_spec(seqs=[(1500, 0), (333, 100)], num_q_heads=8, num_kv_heads=2, page_size=p,
                             config_id=60 + p)
    spec.alpha = 0.3
    full_pipeline(spec)


@pytest.mark.parametrize("g,hkv", [(1, 2), (2, 2), (7, 2), (8, 1), (16, 1)])
def test_group_sizes(g, hkv):
    spec = inputs.small_spec(seqs=[(1100, 37)], num_q_heads=g * hkv, num_kv_heads=hkv, page_size=32,
                             config_id=70 + g, sink=False)
    spec.alpha = 0.25
    full_pipeline(spec)


@pytest.mark.parametrize("seqs", [
    [(1, 0)],                       # one token
    [(128, 127)],                   # one new token after a prefix (decode-like)
    [(129, 0)],                     # ragged by one
    [(127, 0), (1, 0), (256, 255), (640, 512)],
    [(2048, 2047), (300, 0)],
    [(512, 0), (512, 512), (100, 0)],   # a sequence with no new tokens
])
def test_ragged_and_degenerate_batches(seqs):
    spec = inputs.small_spec(seqs=seqs, num_q_heads=4, num_kv_heads=2, page_size=16, config_id=80)
    spec.alpha = 0.4
    full_pipeline(spec)


def test_tiles_with_more_candidates_than_half_the_energy_buffer():
    """The scorer keeps the energies of two consecutive tiles in two halves of one buffer while a separate warp
    selects; a tile with more than 2048 candidate blocks (a sequence beyond 256K tokens) takes the whole buffer
    and must wait for both neighbours.  A chunk of 4096 new tokens behind a 262144-token prefix gives 32 such
    tiles; the short sequences around it give ordinary tiles before and after."""
    spec = inputs.small_spec(seqs=[(700, 0), (266240, 262144), (1000, 0)], num_q_heads=1, num_kv_heads=1,
                             page_size=64, config_id=61)
    spec.alpha = 0.02
    case, dc, wl = make(spec)
    for _ in range(2):   # twice: the second run starts from whatever the first left in shared structures
        dc.select()
        dc.status()
        tot, near = check_lists(dc, wl)
    big = [s for s in wl.segs if s.J_hi + 1 > 2048]
    assert len(big) == 32 and len(wl.segs) > 40
    lists = dc.lists_host()
    dc.sparse()
    dc.status()
    check_attention(dc, wl, lists, dtype=spec.dtype)


def test_scorer_units_pairs_and_singles_of_every_size():
    """The BF16 scorer takes adjacent tiles of a KV head in pairs when the later tile has at most 1024 candidate
    blocks, else one by one (a tile with up to 2048 candidates in its unit's half of the energy buffer, beyond that
    in the whole buffer).  One batch with all three kinds, odd tile counts (a pair cannot straddle two heads or
    sequences) and a ragged last tile; twice, so that the second run meets whatever the first left behind."""
    spec = inputs.small_spec(seqs=[(900, 0), (140000 + 1100, 140000), (1300, 300), (266240 + 700, 266240), (385, 0)],
                             num_q_heads=2, num_kv_heads=2, page_size=64, config_id=62)
    spec.alpha = 0.05
    case, dc, wl = make(spec)
    kinds = {(s.J_hi + 1 > 2048) + (s.J_hi + 1 > 1024) for s in wl.segs}
    assert kinds == {0, 1, 2}
    for _ in range(2):
        dc.select()
        dc.status()
        check_lists(dc, wl)
    lists = dc.lists_host()
    dc.sparse()
    dc.status()
    check_attention(dc, wl, lists, dtype=spec.dtype)


@pytest.mark.parametrize("dtype", ["bf16", "fp8"])
def test_scorer_pairs_beside_single_tiles_with_more_tiles_than_sms(dtype):
    """Tiles are only paired where there are more of them than SMs: the three kinds of unit again with four times the tiles,
    in both data types, odd tile counts and ragged last tiles among them; lists, twice."""
    spec = inputs.small_spec(seqs=[(900, 0), (140000 + 1100, 140000), (1300, 300), (266240 + 700, 266240), (385, 0)],
                             num_q_heads=8, num_kv_heads=2, page_size=64, dtype=dtype, config_id=63)
    spec.alpha = 0.05
    case, dc, wl = make(spec)
    assert dc.plan.num_segments > torch.cuda.get_device_properties(0).multi_processor_count
    for _ in range(2):
        dc.select()
        dc.status()
        check_lists(dc, wl)


@pytest.mark.parametrize("alpha", [0.0, 2.0, 1.0])
def test_alpha_extremes(alpha):
    spec = inputs.small_spec(seqs=[(2000, 0)], num_q_heads=4, num_kv_heads=1, page_size=64, config_id=81, sink=False)
    spec.alpha = alpha
    case, dc, wl = full_pipeline(spec, dense=False)
    cnt = dc.seg_count.cpu().numpy()
    for s in wl.segs:
        if alpha == 0.0:
            assert cnt[s.seg] == s.J_hi + 1
        if alpha == 2.0:
            assert cnt[s.seg] == int(O.forced_mask(s.J_lo, s.J_hi, 128, 256, 512).sum())


def test_truncation_without_correction_and_forced_sets():
    spec = inputs.small_spec(seqs=[(3000, 200)], num_q_heads=8, num_kv_heads=2, page_size=16, config_id=82,
                             sink=False, use_correction=0, sink_tokens=128, window_tokens=0)
    spec.alpha = 0.5
    case, dc, wl = full_pipeline(spec, dense=False)
    assert int(dc.seg_count.sum()) < dc.plan.idx_capacity / 2


def test_correction_changes_the_result_and_matches_oracle():
    """With heavy pruning the corrected output must differ from plain truncation (the term is live)."""
    spec = inputs.small_spec(seqs=[(4096, 0)], num_q_heads=4, num_kv_heads=1, page_size=64, config_id=83,
                             sink=False, sink_tokens=0, window_tokens=0)
    spec.alpha = 2.0                       # forced (diagonal) blocks only
    case, dc, wl = make(spec)
    dc.select(); lists = dc.lists_host()
    dc.sparse(); dc.status()
    check_attention(dc, wl, lists)
    with_corr = dc.out.float().clone()
    case2, dc2, wl2 = make(spec, use_correction=0)
    dc2.select(); dc2.sparse(); dc2.status()
    check_attention(dc2, wl2, dc2.lists_host())
    assert (with_corr - dc2.out.float()).abs().max() > 0.05


def test_caller_supplied_lists_and_recomputed_pooling():
    """Lists need not come from stage 1: feed the oracle's own lists, thinned, into a fresh workspace."""
    spec = inputs.small_spec(seqs=[(2500, 300), (900, 0)], num_q_heads=8, num_kv_heads=2, page_size=32, config_id=84)
    spec.alpha = 0.2
    case, dc, wl = make(spec)
    sel = O.oracle_select(wl)
    rng = np.random.default_rng(0)
    lists = {}
    for s in wl.segs:
        idx = sel[s.seg][0]
        keep = (idx >= s.J_lo) | (rng.random(len(idx)) < 0.6)      # always keep the diagonal band
        lists[s.seg] = idx[keep]
    off = np.array([dc.plan.segment(i)["off"] for i in range(dc.plan.num_segments)] + [dc.plan.idx_capacity])
    cnt = np.array([len(lists[i]) for i in range(dc.plan.num_segments)], dtype=np.int32)
    flat = np.zeros(dc.plan.idx_capacity, dtype=np.int32)
    for i, l in lists.items():
        flat[off[i]:off[i] + len(l)] = l
    dc.seg_offset.copy_(torch.from_numpy(off)); dc.seg_count.copy_(torch.from_numpy(cnt))
    dc.blk_idx.copy_(torch.from_numpy(flat))
    dc.sparse(pooled_valid=False)
    dc.status()
    check_attention(dc, wl, lists)


def test_pooling_as_a_call_of_its_own():
    """fp2_pool_blocks leaves in the workspace exactly what the first kernel of fp2_select_blocks leaves (byte for
    byte), and a following fp2_sparse_prefill with pooled_valid = 1 corrects with it."""
    for dtype in ("bf16", "fp8"):
        spec = inputs.small_spec(seqs=[(2100, 260), (500, 0)], num_q_heads=8, num_kv_heads=2, page_size=32,
                                 config_id=87, dtype=dtype)
        spec.alpha = 0.3
        case, dc, wl = make(spec)
        dc.select(); dc.status()
        ws_after_select = dc.workspace.clone()
        lists = dc.lists_host()
        dc.workspace.zero_()
        dc.pool(); dc.status()
        assert dc.plan.last_launch_count() == 1
        # everything the pooling kernel writes lies before the work-order arrays; compare the pooled region
        pooled = slice(1024, 1024 + 3 * (((sum(-(-lk // 128) for lk, _ in spec.seqs)) * 2 * 128 * 2 + 1023) // 1024 * 1024))
        assert torch.equal(dc.workspace[pooled], ws_after_select[pooled])
        dc.sparse(pooled_valid=True); dc.status()
        check_attention(dc, wl, lists, dtype=dtype)


def test_malformed_lists_are_flagged_not_trapped():
    spec = inputs.small_spec(seqs=[(1000, 0)], num_q_heads=4, num_kv_heads=2, page_size=16, config_id=85)
    case, dc, wl = make(spec)
    dc.select(); dc.status()
    bad = dc.blk_idx.clone()
    bad[int(dc.seg_offset[5])] = 9999            # out of range block id in segment 5
    dc.sparse(blk_idx=bad)
    code, words = dc.status(raise_on_error=False)
    assert code == 1 and words[2] != 0 and words[0] == 0
    dc.sparse()                                   # the context is still usable
    dc.status()
    check_attention(dc, wl, dc.lists_host())


def test_page_ids_outside_the_pool_are_skipped_and_flagged():
    """Stage 1 reads K and V through the page table before any list exists: an id outside [0, num_pages) in a live
    entry must not be dereferenced.  The call is flagged (status word 2, bit 2), nothing traps, and the same
    buffers give the right answer once the table is repaired."""
    spec = inputs.small_spec(seqs=[(1000, 0), (300, 40)], num_q_heads=4, num_kv_heads=2, page_size=16, config_id=86)
    for dtype in ("bf16", "fp8"):
        spec.dtype = dtype
        case, dc, wl = make(spec)
        good = dc.page_table.clone()
        for bad_id in (-1, dc.prm["num_pages"], 2 ** 30):
            dc.page_table.copy_(good)
            dc.page_table[0, 5] = bad_id
            dc.select()
            code, words = dc.status(raise_on_error=False)
            assert code == 1 and (words[2] & 2) and words[0] == 0, (bad_id, code, words)
            dc.sparse()
            code, words = dc.status(raise_on_error=False)
            assert code == 1 and (words[2] & 2) and words[0] == 0, (bad_id, code, words)
        dc.page_table.copy_(good)
        full = dc.select(); dc.status()
        check_lists(dc, wl)
        lists = dc.lists_host()
        dc.sparse(); dc.status()
        check_attention(dc, wl, lists, dtype=dtype)


def test_a_wait_that_runs_out_is_reported_and_leaves_the_context_usable():
    """The library's probe kernel waits, with a budget of a million cycles, on a barrier nobody arrives on.  The wait
    gives up by itself (nothing hangs, nothing traps): FP2_ERR_TIMEOUT with the recorded site, then ordinary calls
    on the same plan and workspace are green."""
    spec = inputs.small_spec(seqs=[(900, 0)], num_q_heads=4, num_kv_heads=2, page_size=16, config_id=88)
    case, dc, wl = make(spec)
    dc.select(); dc.sparse(); dc.status()
    t0 = torch.cuda.Event(enable_timing=True); t1 = torch.cuda.Event(enable_timing=True)
    t0.record()
    binding.fp2_selftest_bounded_wait(dc.plan, dc.workspace)
    t1.record()
    code, words = dc.status(raise_on_error=False)
    assert code == 5, (code, words)                      # FP2_ERR_TIMEOUT
    assert words[0] == 1 and words[1] in (901, 902), words
    assert t0.elapsed_time(t1) < 100.0                   # the budget is under a millisecond of cycles
    code, words = dc.status(raise_on_error=False)        # reading cleared the block
    assert code == 0 and not any(words)
    dc.select(); dc.status()
    check_lists(dc, wl)
    lists = dc.lists_host()
    dc.sparse(); dc.status()
    check_attention(dc, wl, lists)


def test_warps_leave_as_one_after_a_wait_that_ran_out():
    """The probe's lanes give up at different times and leave through the votes, the commit and the CTA barriers that every
    large kernel leaves by; a lane that went its own way would keep the others waiting there.  Several launches in a row, each
    over within its budget (0.5 ms of cycles, 2 ms for copies in flight), each reported."""
    spec = inputs.small_spec(seqs=[(300, 0)], num_q_heads=4, num_kv_heads=2, page_size=16, config_id=89)
    case, dc, wl = make(spec)
    for _ in range(6):
        t0 = torch.cuda.Event(enable_timing=True); t1 = torch.cuda.Event(enable_timing=True)
        t0.record()
        binding.fp2_selftest_bounded_wait(dc.plan, dc.workspace)
        t1.record()
        code, words = dc.status(raise_on_error=False)
        assert code == 5 and words[0] == 1 and words[1] in (901, 902), (code, words)
        assert t0.elapsed_time(t1) < 20.0
    full_pipeline(spec)


def test_two_runs_are_bit_identical():
    spec = inputs.config_spec(2, scale_down=4)
    case, dc, wl = make(spec)
    dc.select(); dc.sparse(); torch.cuda.synchronize()
    a = (dc.blk_idx.clone(), dc.seg_count.clone(), dc.out.clone(), dc.lse.clone())
    dc.out.zero_(); dc.blk_idx.zero_()
    dc.select(); dc.sparse(); torch.cuda.synchronize()
    dc.status()
    assert torch.equal(a[1], dc.seg_count) and torch.equal(a[0], dc.blk_idx)
    assert torch.equal(a[2], dc.out) and torch.equal(a[3], dc.lse)


@pytest.mark.parametrize("dtype", ["bf16", "fp8"])
def test_pooling_in_a_row_uses_the_whole_chip(dtype):
    """A kernel that starts while its predecessor drains may fill a few SMs and leave the others idle: pooling calls in a row took
    twice as long as one behind another kernel.  49 MB of K and V (25 FP8) in a row against the same calls with a kernel of
    torch's, which nothing starts early behind, in between; medians, and a third of slack."""
    import statistics
    spec = inputs.small_spec(seqs=[(12000, 11000)], num_q_heads=8, num_kv_heads=8, page_size=64, dtype=dtype, config_id=91)
    case, dc, wl = make(spec)
    x = torch.zeros(1, device="cuda")

    def time(between, n=60):
        t = []
        for _ in range(9):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda._sleep(2_000_000)               # so that the host is ahead
            e0.record()
            for _ in range(n):
                dc.pool()
                if between:
                    x.add_(1)
            e1.record()
            torch.cuda.synchronize()
            t.append(e0.elapsed_time(e1) / n)
        return statistics.median(t)
    time(False), time(True)
    assert time(False) <= 1.33 * time(True)


def test_launch_counts_are_reported():
    spec = inputs.config_spec(1)
    case, dc, wl = make(spec)
    dc.select()
    assert dc.plan.last_launch_count() == 2           # pool + score/select
    dc.sparse()
    assert dc.plan.last_launch_count() == 4           # order (3) + attention
    dc.plan.set_split(4)
    dc.sparse()
    assert dc.plan.last_launch_count() == 6           # order (3) + split plan + attention + merge


@pytest.mark.parametrize("dtype", ["bf16", "fp8"])
@pytest.mark.parametrize("g", [3, 5, 6, 7, 9, 12])
def test_group_sizes_whose_query_tiles_start_inside_a_box(g, dtype):
    """Group sizes that do not divide 128: a tile starts r0 % g rows into its TMA box (up to 8 for g = 9), with the box's
    overhang on padding; g = 12 is the first whose box of two tiles does not fit and takes the element-wise route.  Ragged
    last tiles, an odd number of tiles (a pair and a single one) and a prefix.  Rows near the start of a sequence put nearly
    all weight on one value, so the bound follows the values: BF16 rounds every probability and the output by at most 2^-8
    of itself, together 2^-7 max |v| (fp32 sums and ex2.approx: well below 1e-3)."""
    spec = inputs.small_spec(seqs=[(700, 0), (1111, 300), (43, 0)], num_q_heads=2 * g, num_kv_heads=2, page_size=16,
                             dtype=dtype, config_id=130 + g)
    spec.alpha = 0.25
    case, dc, wl = make(spec)
    vmax = max(float(np.abs(wl.kv(b, h)[1]).max()) for b in range(3) for h in range(2))
    dc.select()
    dc.status()
    check_lists(dc, wl)
    for lists in (dc.lists_host(), None):
        if lists is not None:
            dc.sparse()
        else:
            dc.dense()
        dc.status()
        Oo, Lo = O.scatter_output(wl, O.oracle_attend(wl, lists, None, dense=lists is None), case.total_q)
        err = np.abs(dc.out.float().cpu().numpy().astype(np.float64) - Oo)[~np.isnan(Oo)]
        assert err.size and err.max() <= vmax * 2.0 ** -7 + 1e-3, (err.max(), vmax)
        gl = dc.lse.cpu().numpy().astype(np.float64)
        ok = ~np.isnan(Lo)
        assert (np.abs(gl - Lo)[ok] / np.maximum(np.abs(Lo[ok]), 1.0)).max() <= TOL_LSE_REL


@pytest.mark.parametrize("n_seg_tokens", [1, 63, 64, 65, 1000])
def test_work_order_takes_every_segment_once(n_seg_tokens):
    """The counting sort behind the attention call: caller lists whose lengths sit on the edges of the sort's classes (0,
    1, 63, 64, 71, 72, 127, 128, 255, 256, 257 blocks), so that a segment dropped or taken twice would leave its rows at the
    poison value or race on them; compared with the dense result of the same rows where the list is complete."""
    lk = 257 * 128
    spec = inputs.small_spec(seqs=[(lk, lk - n_seg_tokens), (300, 0)], num_q_heads=3, num_kv_heads=3, page_size=128,
                             config_id=150)
    case, dc, wl = make(spec, use_correction=0)
    dc.select()
    dc.status()
    off = dc.seg_offset.cpu().numpy()
    edges = [0, 1, 63, 64, 71, 72, 127, 128, 255, 256, 257]
    cnt = np.zeros(dc.plan.num_segments, dtype=np.int32)
    idx = dc.blk_idx.cpu().numpy().copy()
    for s in wl.segs:
        n = min(edges[s.seg % len(edges)], s.J_hi + 1)
        cnt[s.seg] = n
        idx[off[s.seg]:off[s.seg] + n] = np.arange(s.J_hi + 1 - n, s.J_hi + 1)
    dc.sparse(seg_count=torch.from_numpy(cnt).cuda(), blk_idx=torch.from_numpy(idx).cuda())
    dc.status()
    lists = {s.seg: idx[off[s.seg]:off[s.seg] + cnt[s.seg]] for s in wl.segs if cnt[s.seg] > 0}
    check_attention(dc, wl, lists, list(lists))
    assert torch.isfinite(dc.out.float()).all()     # rows without a block come out as zeros


@pytest.mark.parametrize("dtype", ["bf16", "fp8"])
@pytest.mark.parametrize("g", [4, 7, 12])
def test_a_sequence_does_not_depend_on_its_neighbours(g, dtype):
    """The rows behind the end of a sequence in its last tile hold other sequences' queries.  The same sequences with queries of quite
    another size behind them give the same bits: lists, outputs and LSE."""
    spec = inputs.small_spec(seqs=[(701, 100), (333, 0), (915, 700)], num_q_heads=2 * g, num_kv_heads=2, page_size=16,
                             dtype=dtype, config_id=210 + g)
    spec.alpha = 0.2
    res = []
    for loud in (False, True):
        def edit(case):
            if loud:                                   # the second sequence: other queries, a hundred times as large
                a, b = case.cu_seqlens_q.tolist()[1:3]
                if dtype == "fp8":
                    case.q[a:b] = (case.q[a:b].flip(0) & 0x80) | 0x7E
                else:
                    case.q[a:b] = case.q[a:b].flip(0) * 100
        case, dc, wl = make(spec, edit_case=edit)
        dc.select(); dc.sparse(); dc.status()
        sp = dc.out.clone(), dc.lse.clone(), dc.lists_host()
        dc.dense(); dc.status()
        res.append((case.cu_seqlens_q.tolist(), sp, (dc.out.clone(), dc.lse.clone())))
    (cu, (o0, l0, i0), (d0, e0)), (_, (o1, l1, i1), (d1, e1)) = res
    for a, b in ((0, cu[1]), (cu[2], cu[3])):
        assert torch.equal(o0[a:b], o1[a:b]) and torch.equal(l0[:, a:b], l1[:, a:b])
        assert torch.equal(d0[a:b], d1[a:b]) and torch.equal(e0[:, a:b], e1[:, a:b])
    for s in wl.segs:
        if s.b != 1:
            assert np.array_equal(i0[s.seg], i1[s.seg])


@pytest.mark.parametrize("dtype", ["bf16", "fp8"])
@pytest.mark.parametrize("first_loud", [16, 20, 32])
def test_scores_far_above_those_of_the_first_rows(first_loud, dtype):
    """The scorer's exponentials refer to the first 16 rows of a tile; logits more than 2^119 above them must send a batch
    through again.  One KV head, 32 query heads (a tile is 4 tokens), the queries of the heads from first_loud on 64 times as
    large (logits in the hundreds), so that the first batch holds the loudest rows already (with 32 no head is: the plain
    case).  Lists only: probabilities that sharp say nothing more about the attention kernel."""
    spec = inputs.small_spec(seqs=[(5000, 1000), (901, 0)], num_q_heads=32, num_kv_heads=1, page_size=32, dtype=dtype,
                             config_id=160 + first_loud)
    spec.alpha = 0.2

    def louder(case):
        if dtype == "fp8":
            case.q_scale[first_loud:] *= 64
        else:
            case.q[:, first_loud:] *= 64
    case, dc, wl = make(spec, edit_case=louder)
    dc.select()
    dc.status()
    check_lists(dc, wl)


# per row of a tile: by how much its logits (log2) stand above those of the first 16 rows
LOUD = {
    "from16": lambda j: 170.0 if j >= 16 else 0.0,          # first batch, all of it
    "from40": lambda j: 170.0 if j >= 40 else 0.0,          # second batch of 32, first of 64
    "from70": lambda j: 170.0 if j >= 70 else 0.0,          # third, second
    "from100": lambda j: 170.0 if j >= 100 else 0.0,        # the last batch
    "once": lambda j: 170.0 if j == 77 else 0.0,            # one row, the others behind it quiet again
    "stairs": lambda j: 150.0 * (j // 32),                  # every batch of 32, or of 64, once more above the one before
    "stairs64": lambda j: 170.0 * (j // 64) + (90.0 if j % 64 >= 32 else 0.0),   # rises that need a second pass, and rises that do not
}


@pytest.mark.parametrize("dtype,g", [("bf16", 32), ("fp8", 32), ("fp8", 4), ("fp8", 7), ("fp8", 3), ("fp8", 5)])
@pytest.mark.parametrize("shape", list(LOUD))
def test_scores_that_leave_the_reference_behind_in_a_given_batch(shape, dtype, g):
    """The scorer goes through a tile's 128 rows in batches (64; FP8 with row multipliers in shared memory, here groups of 32: 32)
    against the maximum of the first 16, and a batch that comes out above 2^119 is done again against its own maximum, the sum so
    far scaled down.  Here one dimension of every key holds a constant c and the queries' entry there sets a row's level, so which
    batches that happens in is known: asserted from the oracle's logits.  Groups of 32: a tile is 4 tokens x 32 heads; pairs, a
    single tile, and a last tile of 3 tokens.  Smaller groups: single tiles, a last one of a few rows.  No block is forced into a
    list."""
    spec = inputs.small_spec(seqs=[(5000, 4001), (902, 3)], num_q_heads=g, num_kv_heads=1, page_size=32, dtype=dtype,
                             config_id=200, locality_a=0.5)
    spec.alpha = 0.3

    def levels(case):
        c = 128.0 * float(case.k_scale[0]) if dtype == "fp8" else 2.0
        case.k_cache[..., 0] = 0x70 if dtype == "fp8" else c
        if dtype == "fp8":
            q = case.q.view(torch.float8_e4m3fn).float() * case.q_scale[None, :, None]
        else:
            q = case.q.float()
        cu = case.cu_seqlens_q.tolist()
        for b in range(2):
            r = torch.arange((cu[b + 1] - cu[b]) * g)
            lv = torch.tensor([LOUD[shape](int(j) % 128) for j in r])
            q[cu[b]:cu[b + 1], :, 0] = (lv / (c * 128 ** -0.5 * np.log2(np.e))).view(-1, g)
        if dtype == "fp8":
            case.q_scale[:] = q.abs().amax() / 448.0
            case.q[:] = inputs.quantize_e4m3(q, case.q_scale[None, :, None])
        else:
            case.q[:] = q.to(torch.bfloat16)
    case, dc, wl = make(spec, edit_case=levels, sink_tokens=0, window_tokens=0)
    W = 32 if dtype == "fp8" and g == 32 else 64
    redone = {}
    for s in wl.segs:
        x = O.tile_queries(wl.q_seq(s.b), wl.p, s) @ wl.kv(s.b, s.h)[2][:s.J_hi + 1].T * wl.p.scale * np.log2(np.e)
        ref = x[:16].max(axis=0)                        # per block
        for k in range(0, x.shape[0], W):
            top = x[k:k + W].max(axis=0)
            up = top - ref > 120.0
            assert (up | (top - ref < 112.0)).all()     # 2^119.6 is the limit on a sum of up to 128: none is near it
            redone.setdefault(k // W, []).append(up)
            ref = np.where(up, np.maximum(top, ref), ref)
    redone = {k: bool(np.concatenate(v).any()) for k, v in redone.items()}
    want = {"from16": [0], "from40": [40 // W], "from70": [70 // W], "from100": [100 // W], "once": [77 // W],
            "stairs": [1, 2, 3] if W == 32 else [0, 1], "stairs64": [2] if W == 32 else [1]}[shape]
    assert [k for k in sorted(redone) if redone[k]] == list(want), redone
    dc.select()
    dc.status()
    tot, _ = check_lists(dc, wl)
    assert 0.1 < tot / dc.plan.idx_capacity < 0.9


@pytest.mark.parametrize("dtype", ["bf16", "fp8"])
@pytest.mark.parametrize("quiet", [16, 31])
def test_scores_whose_first_rows_are_below_the_range_of_fp32(quiet, dtype):
    """The scorer takes its reference from the first 16 rows of a tile.  Where all of their logits overflow to -inf (heads 0 .. 15
    query one dimension with -3e38, in which every key is positive), they contribute nothing and the other rows' energies
    decide, as they do in exact arithmetic.  Whole and partial tiles, pairs and a single tile; no block is forced into a list,
    and the threshold divides the candidates."""
    spec = inputs.small_spec(seqs=[(5000, 4001), (901, 0)], num_q_heads=32, num_kv_heads=1, page_size=32, dtype=dtype,
                             config_id=190, locality_a=0.5)
    spec.alpha = 0.3

    def lowest(case):
        if dtype == "fp8":
            case.k_cache[..., 0] = 0x70                 # 128 in raw units
            case.q[:, :quiet] = 0
            case.q[:, :quiet, 0] = 0xFE                 # -448
            case.q_scale[:quiet] = 1e38
        else:
            case.k_cache[..., 0] = 16.0
            case.q[:, :quiet] = 0
            case.q[:, :quiet, 0] = -3e38
    case, dc, wl = make(spec, edit_case=lowest, sink_tokens=0, window_tokens=0)
    qt = O.tile_queries(wl.q_seq(0), wl.p, wl.segs[0])
    s = qt @ wl.kv(0, 0)[2].T * wl.p.scale * np.log2(np.e)
    assert s[:quiet].max() < -3.5e38 and np.abs(s[quiet:32]).max() < 1e4
    dc.select()
    dc.status()
    tot, _ = check_lists(dc, wl)
    assert 0.1 < tot / dc.plan.idx_capacity < 0.9


@pytest.mark.parametrize("hkv", [1, 3])
def test_work_order_with_a_few_long_segments(hkv):
    """More segments than workers times eight, so that only some count as long and go first: lists of 0 to 2 blocks (the limit
    lies between 1 and 2), every 13th with 3, every 101st complete.  A segment dropped by either part of the order would
    leave its rows at the poison value."""
    spec = inputs.small_spec(seqs=[(3300 if hkv == 3 else 9900, 0)], num_q_heads=32 * hkv, num_kv_heads=hkv, page_size=128,
                             config_id=152 + hkv)
    case, dc, wl = make(spec, use_correction=0)
    dc.select()
    dc.status()
    off = dc.seg_offset.cpu().numpy()
    cnt = np.zeros(dc.plan.num_segments, dtype=np.int32)
    idx = dc.blk_idx.cpu().numpy().copy()
    for s in wl.segs:
        n = s.J_hi + 1 if s.seg % 101 == 0 else min(3 if s.seg % 13 == 0 else s.seg % 3, s.J_hi + 1)
        cnt[s.seg] = n
        idx[off[s.seg]:off[s.seg] + n] = np.arange(s.J_hi + 1 - n, s.J_hi + 1)
    workers = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    assert 1.0 < cnt.sum() / (8 * workers) < 2.0
    dc.sparse(seg_count=torch.from_numpy(cnt).cuda(), blk_idx=torch.from_numpy(idx).cuda())
    dc.status()
    some = [s.seg for s in wl.segs if cnt[s.seg] > 0 and (s.seg % 101 == 0 or s.seg % 97 == 0)]
    check_attention(dc, wl, {s: idx[off[s]:off[s] + cnt[s]] for s in some}, some)
    assert torch.isfinite(dc.out.float()).all()


@pytest.mark.parametrize("hkv", [8192, 8193, 12300])
def test_work_order_of_very_many_heads(hkv):
    """The order's per-head counts are in shared memory up to 8192 KV heads; more than about 11700 would not fit.  Beyond, the order
    is KV-head-major without them.  One query head per KV head, nine tokens in two pages; dense against fp32 attention
    (tolerance as for the oracle)."""
    n = 9
    prm = dict(num_seqs=1, total_q=n, num_q_heads=hkv, num_kv_heads=hkv, head_dim=128, block_size=128, tile_rows=128,
               page_size=8, num_pages=3, max_pages_per_seq=2, sink_tokens=256, window_tokens=512, use_correction=1,
               alpha=0.1, softmax_scale=0.0, dtype=0)
    plan = binding.Plan(prm, [0, n], [n])
    g = torch.Generator(device="cuda").manual_seed(hkv)
    q, k, v = (torch.randn(*s, hkv, 128, generator=g, device="cuda").to(torch.bfloat16) for s in ((n,), (3, 8), (3, 8)))
    pt = torch.tensor([[2, 0]], dtype=torch.int32, device="cuda")
    cu = torch.tensor([0, n], dtype=torch.int32, device="cuda")
    lk = torch.tensor([n], dtype=torch.int32, device="cuda")
    ws = plan.new_workspace()
    out = torch.full((n, hkv, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.full((hkv, n), float("nan"), device="cuda")
    binding.fp2_dense_prefill(plan, q, k, v, pt, cu, lk, None, None, None, out, lse, ws)
    binding.fp2_read_status(plan, ws)
    K, V = (torch.cat([x[2], x[0]])[:n].float() for x in (k, v))
    s = torch.einsum("ihd,jhd->hij", q.float(), K) / 128 ** 0.5
    s = s.masked_fill(torch.ones(n, n, dtype=torch.bool, device="cuda").triu(1), float("-inf"))
    ref = torch.einsum("hij,jhd->ihd", s.softmax(-1), V)
    vmax = V.abs().max().item()                    # P and the output each round by 2^-9 of a value: 2^-7 vmax holds both
    assert (out.float() - ref).abs().max().item() <= vmax * 2.0 ** -7 + 1e-3
    assert (lse - torch.logsumexp(s, -1)).abs().max().item() <= TOL_LSE_REL
    plan.close()


@pytest.mark.parametrize("p,hkv,seqs", [
    (8, 2, [(3000, 0), (130, 2)]),           # ragged last pages, two sequences
    (128, 2, [(3200, 100)]),                 # whole blocks
    (32, 3, [(1, 0), (2900, 0), (257, 256)]),  # a head count that no power of two divides, a one-token sequence
])
def test_fp8_values_widened_once_per_call(p, hkv, seqs):
    """FP8 calls with enough iterations (4000 + 7 per block and KV head) read V as an F16 copy in the workspace; shorter ones
    widen every tile in the kernel.  Both routes against the oracle, sparse and dense, at ragged lengths and the smallest
    and largest page; and a page id outside the pool is still flagged on the copying route."""
    spec = inputs.small_spec(seqs=seqs, num_q_heads=8 * hkv, num_kv_heads=hkv, page_size=p, dtype="fp8",
                             config_id=160 + p)
    spec.alpha = 0.05
    case, dc, wl = full_pipeline(spec)
    assert dc.plan.idx_capacity >= 4000 + 7 * hkv * sum(-(-lk // 128) for lk, _ in seqs)
    small = inputs.small_spec(seqs=[(400, 0)], num_q_heads=8 * hkv, num_kv_heads=hkv, page_size=p, dtype="fp8", config_id=170)
    small.alpha = 0.05
    _, dcs, _ = full_pipeline(small)
    assert dcs.plan.idx_capacity < 4000
    good = dc.page_table.clone()
    dc.page_table[len(seqs) - 1, 0] = dc.prm["num_pages"] + 3
    dc.dense()
    code, words = dc.status(raise_on_error=False)
    assert code == 1 and words[2] & 2
    dc.page_table.copy_(good)

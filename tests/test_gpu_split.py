"""KV splitting (Eq. 18): the attention path with segments cut into parts and merged must give the oracle's
result within the same gates, whatever the number of parts."""
import numpy as np
import pytest
import torch

from oracle import fp2_oracle as O
from paper_2608_19758_b200 import binding, inputs
from test_gpu_parity import check_attention, check_lists, make

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("target", [1, 2, 5, 0, -1])
@pytest.mark.parametrize("dtype,g,hkv,p,seqs", [
    ("bf16", 4, 2, 16, [(1500, 300), (700, 0), (129, 128), (40, 0)]),
    ("bf16", 7, 1, 64, [(3000, 0)]),
    ("fp8", 4, 2, 32, [(2500, 500), (257, 0)]),
])
def test_split_attention_matches_oracle(target, dtype, g, hkv, p, seqs):
    spec = inputs.small_spec(seqs=seqs, num_q_heads=g * hkv, num_kv_heads=hkv, page_size=p, dtype=dtype,
                             config_id=70 + g)
    spec.alpha = 0.2
    case, dc, wl = make(spec)
    dc.plan.set_split(target)
    dc.select(); dc.status()
    lists = dc.lists_host()
    dc.sparse(); dc.status()
    if target != 0:                                    # automatic: the host may see that nothing can be split
        assert dc.plan.last_launch_count() == (4 if target < 0 else 6)
    check_attention(dc, wl, lists, dtype=dtype)
    dc.dense(); dc.status()
    check_attention(dc, wl, None, dense=True, dtype=dtype)


def test_split_without_correction_and_with_caller_lists():
    """Lists of one block per segment (every part but the first is empty at target 1 ... no: one iteration, one
    part) and long hand-made lists that are cut into many parts."""
    spec = inputs.small_spec(seqs=[(4096, 0)], num_q_heads=4, num_kv_heads=2, page_size=64, config_id=77)
    case, dc, wl = make(spec, use_correction=0)
    dc.plan.set_split(1)
    dc.select(); dc.status()
    off = dc.seg_offset.cpu().numpy()
    cnt = np.zeros(dc.plan.num_segments, dtype=np.int32)
    idx = dc.blk_idx.cpu().numpy().copy()
    lists = {}
    for s in wl.segs:                                   # every second candidate, always the diagonal band
        L = sorted(set(range(0, s.J_hi + 1, 2)) | set(range(s.J_lo, s.J_hi + 1)))
        lists[s.seg] = np.asarray(L, dtype=np.int32)
        cnt[s.seg] = len(L)
        idx[off[s.seg]:off[s.seg] + len(L)] = L
    dc.sparse(seg_count=torch.from_numpy(cnt).cuda(), blk_idx=torch.from_numpy(idx).cuda())
    dc.status()
    check_attention(dc, wl, lists)


def test_split_is_deterministic_and_equals_unsplit_within_rounding():
    spec = inputs.config_spec(1)
    case, dc, wl = make(spec)
    dc.select(); dc.status()
    dc.plan.set_split(2)
    dc.sparse(); torch.cuda.synchronize()
    a, la = dc.out.clone(), dc.lse.clone()
    dc.sparse(); torch.cuda.synchronize()
    assert torch.equal(a, dc.out) and torch.equal(la, dc.lse)
    dc.plan.set_split(-1)
    dc.sparse(); torch.cuda.synchronize()
    dc.status()
    assert (a.float() - dc.out.float()).abs().max().item() <= 2e-2
    assert torch.allclose(la, dc.lse, rtol=1e-5, atol=1e-5)


@pytest.mark.parametrize("target", [0, 1, 100000])
def test_a_split_request_that_does_not_apply_leaves_the_cutting_on(target):
    """Plans of 4 to 16 segments per worker are never split on request, and a part of 100000 iterations fits nothing; such calls are
    what they are by default: segments longer than a worker's share are cut, with the same launches and the same bits.  One
    page for all tokens keeps the cache small."""
    workers = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    n_seg = 4 * workers + 16 if target < 100000 else 40
    hq, lk = 64, 520 * 128
    lq = 2 * n_seg                                       # 64 heads on one: 2 tokens per tile
    prm = dict(num_seqs=1, total_q=lq, num_q_heads=hq, num_kv_heads=1, head_dim=128, block_size=128, tile_rows=128,
               page_size=128, num_pages=4, max_pages_per_seq=520, sink_tokens=256, window_tokens=512, use_correction=1,
               alpha=0.1, softmax_scale=0.0, dtype=0)
    plan = binding.Plan(prm, [0, lq], [lk])
    assert plan.num_segments == n_seg
    g = torch.Generator(device="cuda").manual_seed(3)
    q, k, v = (torch.randn(*s, 128, generator=g, device="cuda").to(torch.bfloat16)
               for s in ((lq, hq), (4, 128, 1), (4, 128, 1)))
    pt = (torch.arange(520, device="cuda") % 4).to(torch.int32)[None]
    cu = torch.tensor([0, lq], dtype=torch.int32, device="cuda")
    lk_t = torch.tensor([lk], dtype=torch.int32, device="cuda")
    ws = plan.new_workspace()
    off, cnt, idx = plan.new_lists()
    binding.fp2_select_blocks(plan, q, k, v, pt, cu, lk_t, None, None, None, off, cnt, idx, ws)
    # every 40th list complete: far above a worker's share
    o, c, i = off.cpu(), cnt.cpu(), idx.cpu()
    for s in range(n_seg):
        d = plan.segment(s)
        first = 0 if s % 40 == 7 else d["J_hi"] - 6
        c[s] = d["J_hi"] + 1 - first
        i[int(o[s]):int(o[s]) + int(c[s])] = torch.arange(first, d["J_hi"] + 1, dtype=torch.int32)
    assert int(c.max()) >= 500 and int(c.max()) > int(c.sum()) / workers
    cnt, idx = c.cuda(), i.cuda()

    def run():
        out = torch.full((lq, hq, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((hq, lq), float("nan"), device="cuda")
        binding.fp2_sparse_prefill(plan, q, k, v, pt, cu, lk_t, off, cnt, idx, None, None, None, out, lse, ws)
        binding.fp2_read_status(plan, ws)
        return out, lse, plan.last_launch_count()
    o0, l0, n0 = run()
    plan.set_split(target)
    o1, l1, n1 = run()
    assert n0 == n1 == 5
    assert torch.equal(o0, o1) and torch.equal(l0, l1)


def test_large_plans_are_not_split():
    spec = inputs.config_spec(2, scale_down=2)           # 16K tokens: 4096 segments, more than 4 per worker
    case, dc, wl = make(spec)
    dc.plan.set_split(1)
    dc.select(); dc.sparse(); dc.status()
    assert dc.plan.last_launch_count() == 4


@pytest.mark.parametrize("dtype,g,hkv,seqs", [
    ("bf16", 4, 1, [(66000, 65700), (9000, 8000), (129, 0)]),    # ragged last tiles
    ("bf16", 7, 1, [(70000, 69300)]),
    ("fp8", 4, 2, [(66000, 65500), (5000, 4000)]),
])
def test_longest_segments_are_cut_without_being_asked(dtype, g, hkv, seqs):
    """Caller lists: every 9th segment complete (500 blocks and more, above a worker's share), the others the diagonal band.
    The attention call cuts the long ones into parts and merges them (one launch more).  The second run equals the first bit
    for bit; dense, where all segments of the long sequence are that long, and more of them than partial results fit."""
    spec = inputs.small_spec(seqs=seqs, num_q_heads=g * hkv, num_kv_heads=hkv, page_size=64, dtype=dtype, config_id=180 + g)
    case, dc, wl = make(spec)
    dc.select(); dc.status()
    off = dc.seg_offset.cpu().numpy()
    cnt = np.zeros(dc.plan.num_segments, dtype=np.int32)
    idx = dc.blk_idx.cpu().numpy().copy()
    for s in wl.segs:
        first = 0 if s.seg % 9 == 0 else s.J_lo
        cnt[s.seg] = s.J_hi + 1 - first
        idx[off[s.seg]:off[s.seg] + cnt[s.seg]] = np.arange(first, s.J_hi + 1)
    workers = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    assert cnt.max() >= 500 and cnt.max() > cnt.sum() / workers
    lists = {s.seg: idx[off[s.seg]:off[s.seg] + cnt[s.seg]] for s in wl.segs}
    c, i = torch.from_numpy(cnt).cuda(), torch.from_numpy(idx).cuda()
    dc.sparse(seg_count=c, blk_idx=i); dc.status()
    assert dc.plan.last_launch_count() == 5
    check_attention(dc, wl, lists, dtype=dtype)
    o, l = dc.out.clone(), dc.lse.clone()
    dc.sparse(seg_count=c, blk_idx=i); dc.status()
    assert torch.equal(o, dc.out) and torch.equal(l, dc.lse)
    dc.dense(); dc.status()
    check_attention(dc, wl, None, dense=True, dtype=dtype)

"""The decode entry point that allocates nothing (fnpu_decode_attn_noalloc).

It exists for callers that may not call cudaMalloc (code confined to memory
another framework reserved, or a process whose device memory is fixed at
start): it keeps its split scratch in a fixed array inside the library. These
tests call it through the C ABI, twice in a row where it matters, and check
the results against the fp64 oracle and against the planned path
(fnpu_mixed_attn_plan + fnpu_mixed_attn_run) on the same decode batch, within
the parity tolerances used by the other GPU tests. One test feeds it a context
longer than the bound it was given and a block id outside the pool, laid out
so that even an unchecked read would stay inside allocated memory, and checks
that the kernel skips them and raises the device error flag.

The file is collected last and also passes on its own in a fresh process.
"""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

O_TOL = 2e-2
LSE_TOL = 1e-3


def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _oracle_after_append(batch):
    ref_o, ref_l, _, _ = oracle.run_step(batch)
    return ref_o, ref_l


@pytest.mark.parametrize("split_keys", [0, 256])
def test_noalloc_decode_matches_oracle_and_planned_path_twice(split_keys):
    _need_gpu()
    import paper_2606_04415_gb300 as fnpu
    from paper_2606_04415_gb300.step import DeviceStep

    batch = W.make_batch("qwen_decode", seed=3)
    st = DeviceStep(batch)
    st.run()  # append + planned attention
    plan_o, plan_l = st.results()
    ref_o, ref_l = _oracle_after_append(batch)

    ctx = torch.from_numpy(batch.context_len).cuda()
    bt = torch.from_numpy(batch.block_table).cuda()
    T, Hq, D = st.out.shape
    for call in range(2):
        out = torch.full((T, Hq, D), float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((T, Hq), float("nan"), dtype=torch.float32, device="cuda")
        fnpu.decode_attn_noalloc(st.desc, ctx, bt, int(batch.context_len.max()), st.q, st.k_cache,
                                 st.v_cache, out, lse, split_keys=split_keys)
        torch.cuda.synchronize()
        o = out.float().cpu().numpy()
        l = lse.cpu().numpy()
        assert np.isfinite(o).all() and np.isfinite(l).all(), f"call {call}"
        assert np.abs(o - ref_o).max() <= O_TOL, f"call {call}: oracle"
        assert np.abs(l - ref_l).max() <= LSE_TOL, f"call {call}: oracle"
        assert np.abs(o - plan_o).max() <= O_TOL, f"call {call}: planned path"
        assert np.abs(l - plan_l).max() <= LSE_TOL, f"call {call}: planned path"
    assert fnpu.check() == fnpu.FNPU_OK


def test_noalloc_decode_d64_partial_group_single_and_multi_split():
    """head_dim 64 with 3 query heads per kv head (the 8 MMA columns only
    partly filled); contexts from 1 key up to and past one split, so that
    single-split sequences (written directly) and split ones (merged from their
    partials) both occur, checked against the oracle and the
    planned path on two calls in a row."""
    _need_gpu()
    import paper_2606_04415_gb300 as fnpu
    from paper_2606_04415_gb300.step import DeviceStep

    shape = W.Shape(6, 2, 64, 64, 16, False)
    ctx = np.array([1, 2, 15, 16, 17, 63, 64, 65, 127, 128, 129, 200, 255, 256, 257, 300], np.int32)
    rng = np.random.default_rng(41)
    batch = W.build_batch(shape, np.ones_like(ctx), ctx, np.ones(len(ctx), np.uint8), rng, name="noalloc_d64")
    st = DeviceStep(batch)
    st.run()
    plan_o, plan_l = st.results()
    ref_o, ref_l = _oracle_after_append(batch)

    dctx = torch.from_numpy(batch.context_len).cuda()
    bt = torch.from_numpy(batch.block_table).cuda()
    T, Hq, D = st.out.shape
    for call in range(2):
        out = torch.full((T, Hq, D), float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((T, Hq), float("nan"), dtype=torch.float32, device="cuda")
        fnpu.decode_attn_noalloc(st.desc, dctx, bt, int(ctx.max()), st.q, st.k_cache, st.v_cache, out, lse,
                                 split_keys=128)
        torch.cuda.synchronize()
        o = out.float().cpu().numpy()
        l = lse.cpu().numpy()
        assert np.isfinite(o).all() and np.isfinite(l).all(), f"call {call}"
        assert np.abs(o - ref_o).max() <= O_TOL, f"call {call}: oracle"
        assert np.abs(l - ref_l).max() <= LSE_TOL, f"call {call}: oracle"
        assert np.abs(o - plan_o).max() <= O_TOL, f"call {call}: planned path"
        assert np.abs(l - plan_l).max() <= LSE_TOL, f"call {call}: planned path"
    assert fnpu.check() == fnpu.FNPU_OK


def test_noalloc_rejects_requests_beyond_its_scratch():
    _need_gpu()
    import paper_2606_04415_gb300 as fnpu
    desc = fnpu.make_desc(28, 4, 128, 128, 16, 1 << 20)
    n = 4096
    ctx = torch.full((n,), 16384, dtype=torch.int32, device="cuda")
    bt = torch.zeros((n, 1024), dtype=torch.int32, device="cuda")
    dummy = torch.zeros(16, dtype=torch.bfloat16, device="cuda")
    with pytest.raises(fnpu.FnpuError) as e:
        fnpu.decode_attn_noalloc(desc, ctx, bt, 16384, dummy, dummy, dummy, dummy, dummy.float(),
                                 split_keys=64)
    assert e.value.code == fnpu.FNPU_EINVAL


def test_noalloc_skips_and_flags_out_of_range_context_and_block():
    """Sequence 1's context exceeds the max_context_len the call was given and
    sequence 2's block table names a block past desc.num_blocks. The buffers are
    laid out so that neither would leave allocated memory even unchecked: the
    block table is wide enough for the longer context, and the pools hold 8
    blocks more than the descriptor declares. The kernel must skip both (no
    write to sequence 1's rows), raise the flag, and leave the other sequences
    right."""
    _need_gpu()
    import paper_2606_04415_gb300 as fnpu

    shape = W.Shape(6, 2, 64, 64, 16, False)
    ctx = np.array([40, 100, 70, 33], np.int32)
    rng = np.random.default_rng(7)
    batch = W.build_batch(shape, np.ones_like(ctx), ctx, np.ones(len(ctx), np.uint8), rng, name="noalloc_guard",
                          extra_bt_cols=8)
    # reference on the appended cache, before the bad inputs are made
    ref_o, ref_l = _oracle_after_append(batch)
    kc = oracle.kv_append(batch.k_cache, batch.k_new, batch.slot_mapping)
    vc = oracle.kv_append(batch.v_cache, batch.v_new, batch.slot_mapping)
    nb = batch.num_blocks
    pad = np.zeros((8,) + kc.shape[1:], np.uint16)  # 8 allocated blocks past the declared pool
    k_pool = torch.from_numpy(np.concatenate([kc, pad]).view(np.int16)).cuda().view(torch.bfloat16)
    v_pool = torch.from_numpy(np.concatenate([vc, pad]).view(np.int16)).cuda().view(torch.bfloat16)
    q = torch.from_numpy(batch.q.view(np.int16)).cuda().view(torch.bfloat16)
    desc = fnpu.make_desc(6, 2, 64, 64, 16, nb)

    max_ctx = 80           # sequence 1 (100 keys) is beyond it
    bt = batch.block_table.copy()
    assert bt.shape[1] * 16 >= 100  # its row still covers 100 keys
    bt[2, 1] = nb + 3      # sequence 2: a block id past the declared pool, inside the allocation
    dctx = torch.from_numpy(ctx).cuda()
    dbt = torch.from_numpy(bt).cuda()
    T, Hq = len(ctx), 6
    out = torch.full((T, Hq, 64), float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.full((T, Hq), float("nan"), dtype=torch.float32, device="cuda")
    fnpu.decode_attn_noalloc(desc, dctx, dbt, max_ctx, q, k_pool, v_pool, out, lse, split_keys=64)
    assert fnpu.check() == fnpu.FNPU_EDEVICE_RANGE
    assert fnpu.check() == fnpu.FNPU_OK  # read and cleared
    o = out.float().cpu().numpy()
    l = lse.cpu().numpy()
    assert np.isnan(o[1]).all() and np.isnan(l[1]).all()  # skipped: left as it was
    for s in (0, 3):
        assert np.abs(o[s] - ref_o[s]).max() <= O_TOL
        assert np.abs(l[s] - ref_l[s]).max() <= LSE_TOL


@pytest.mark.parametrize("bs", [16, 48, 24])
@pytest.mark.parametrize("heads", [(8, 8), (9, 3), (35, 5), (28, 4)])
@pytest.mark.parametrize("split_keys", [0, 64])
def test_noalloc_head_groups_block_sizes_and_split_lengths(heads, bs, split_keys):
    """One, several and a ragged last group of kv heads; block sizes on the
    TMA-fed path and (24) off it; contexts at split and stage edges, one of
    them the bound itself, with open and given split lengths."""
    _need_gpu()
    import paper_2606_04415_gb300 as fnpu
    from paper_2606_04415_gb300.step import DeviceStep
    hq, hkv = heads
    sh = W.Shape(hq, hkv, 128, 128, bs, False)
    ctx = [1, 16, 17, 63, 64, 65, 128, 129, 512, 513, 1300]
    rng = np.random.default_rng(10 * hkv + bs)
    batch = W.build_batch(sh, [1] * len(ctx), ctx, [1] * len(ctx), rng, name="noalloc_groups")
    st = DeviceStep(batch)
    st.append()
    out = torch.full_like(st.out, float("nan"))
    lse = torch.full_like(st.lse, float("nan"))
    fnpu.decode_attn_noalloc(st.desc, torch.from_numpy(batch.context_len).cuda(), torch.from_numpy(batch.block_table).cuda(),
                             1300, st.q, st.k_cache, st.v_cache, out, lse, split_keys=split_keys)
    torch.cuda.synchronize()
    assert fnpu.check() == fnpu.FNPU_OK
    ref_o, ref_l = _oracle_after_append(batch)
    assert np.abs(out.float().cpu().numpy() - ref_o).max() <= O_TOL
    assert np.abs(lse.cpu().numpy() - ref_l).max() <= LSE_TOL


@pytest.mark.parametrize("dim", [64, 128])
def test_noalloc_many_sequences_of_a_stage_or_three(dim):
    """Several items a CTA, most of one 16-key stage (as the planned decode's test
    of the item ring): every row right, and the same bits again."""
    _need_gpu()
    import paper_2606_04415_gb300 as fnpu
    from paper_2606_04415_gb300.step import DeviceStep
    sh = W.Shape(4, 2, dim, dim, 16, False)
    rng = np.random.default_rng(dim + 1)
    ctx = np.concatenate([rng.integers(33, 49, size=400), rng.integers(1, 17, size=3000)])
    batch = W.build_batch(sh, np.ones_like(ctx), ctx, np.ones(len(ctx), np.uint8), rng, name="noalloc_short")
    st = DeviceStep(batch)
    st.append()
    ref_o, ref_l = _oracle_after_append(batch)
    dctx, bt = torch.from_numpy(batch.context_len).cuda(), torch.from_numpy(batch.block_table).cuda()
    first = None
    for call in range(5):
        out, lse = torch.full_like(st.out, float("nan")), torch.full_like(st.lse, float("nan"))
        fnpu.decode_attn_noalloc(st.desc, dctx, bt, 48, st.q, st.k_cache, st.v_cache, out, lse)
        torch.cuda.synchronize()
        o, l = out.float().cpu().numpy(), lse.cpu().numpy()
        if first is None:
            first = o, l
            assert np.abs(o - ref_o).max() <= O_TOL and np.abs(l - ref_l).max() <= LSE_TOL
        assert np.array_equal(o, first[0]) and np.array_equal(l, first[1]), f"call {call}"
    assert fnpu.check() == fnpu.FNPU_OK


@pytest.mark.parametrize("heads,dim", [((32, 8), 128), ((28, 4), 128), ((4, 2), 64)])
def test_noalloc_probabilities_lose_nothing_to_bf16(heads, dim):
    """As the planned decode's test of the same name: a result is off by little
    more than its own rounding to bf16."""
    _need_gpu()
    import paper_2606_04415_gb300 as fnpu
    from paper_2606_04415_gb300.step import DeviceStep
    sh = W.Shape(*heads, dim, dim, 16, False)
    ctx = [700, 1500, 333, 2048, 64]
    batch = W.build_batch(sh, [1] * len(ctx), ctx, [1] * len(ctx), np.random.default_rng(dim), name="fine_p")
    st = DeviceStep(batch)
    st.append()
    fnpu.decode_attn_noalloc(st.desc, torch.from_numpy(batch.context_len).cuda(), torch.from_numpy(batch.block_table).cuda(),
                             max(ctx), st.q, st.k_cache, st.v_cache, st.out, st.lse)
    out, _ = st.results()
    ref, _ = _oracle_after_append(batch)
    rounded = W.bf16_bits_to_f32(W.f32_to_bf16_bits(ref))
    assert np.linalg.norm(out - ref) <= 1.05 * np.linalg.norm(rounded - ref)


_ONE_CALL_PREPARES = """
import torch
import paper_2606_04415_gb300 as fnpu

def call(n, ctx, hq, hkv, d, bs=16):
    nb = n * ((ctx + bs - 1) // bs)
    desc = fnpu.make_desc(hq, hkv, d, d, bs, nb)
    cl = torch.full((n,), ctx, dtype=torch.int32, device="cuda")
    bt = torch.arange(nb, dtype=torch.int32, device="cuda").view(n, -1)
    q = torch.randn(n, hq, d, device="cuda").bfloat16()
    k, v = (torch.randn(nb, bs, hkv, d, device="cuda").bfloat16() for _ in range(2))
    out, lse = torch.empty_like(q), torch.empty(n, hq, device="cuda")
    return (lambda: fnpu.decode_attn_noalloc(desc, cl, bt, ctx, q, k, v, out, lse)), out, lse

small = call(1, 16, 4, 2, 64, 24)
others = [call(n, ctx, hq, hkv, d, bs) for hq, hkv, d, bs in
          [(32, 8, 128, 16), (9, 3, 128, 16), (4, 4, 64, 16), (6, 2, 64, 16), (28, 4, 128, 24), (4, 4, 64, 24)]
          for n, ctx in [(1, 60), (1, 5000), (20, 2000), (60, 4000)]]
torch.cuda.synchronize()
small[0]()
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
for f, out, lse in others[::2]:
    f()
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free
for f, out, lse in others:
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        f()
    g.replay()
    torch.cuda.synchronize()
    a = out.clone(), lse.clone()
    out.fill_(float("nan"))
    lse.fill_(float("nan"))
    f()
    torch.cuda.synchronize()
    assert torch.equal(a[0], out) and torch.equal(a[1], lse)
    assert torch.isfinite(out).all() and torch.isfinite(lse).all()
assert fnpu.check() == fnpu.FNPU_OK
print("prepared")
"""


def test_noalloc_one_call_prepares_all_later_ones():
    """In a fresh process, one small call; after it no call takes device memory,
    and every other head shape, ring depth and merge (half of them not called
    before) is captured into a graph and replayed, with a direct call's results."""
    _need_gpu()
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _ONE_CALL_PREPARES], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "prepared" in r.stdout, r.stdout + r.stderr


@pytest.mark.parametrize("hkv,share,bound", [(1, 0.75, 700), (2, 2.0, 512), (2, 2.0, 511)])
def test_noalloc_narrow_heads_on_both_sides_of_the_kernels_line(hkv, share, bound):
    """One or two 64-wide kv heads: up to 3/4 of a sequence per SM (one head), or
    fewer than two with bounds from 512 keys on (two heads), the TMA kernel runs,
    beyond it the per-head one."""
    _need_gpu()
    import paper_2606_04415_gb300 as fnpu
    from paper_2606_04415_gb300.step import DeviceStep
    line = int(share * torch.cuda.get_device_properties(0).multi_processor_count)
    for n in (line - 1, line, line + 1):
        rng = np.random.default_rng(n)
        ctx = rng.integers(1, bound + 1, size=n)
        ctx[0] = bound
        batch = W.build_batch(W.Shape(4, hkv, 64, 64, 16, False), [1] * n, ctx, [1] * n, rng, name="noalloc_narrow")
        st = DeviceStep(batch)
        st.append()
        fnpu.decode_attn_noalloc(st.desc, torch.from_numpy(batch.context_len).cuda(), torch.from_numpy(batch.block_table).cuda(),
                                 bound, st.q, st.k_cache, st.v_cache, st.out, st.lse)
        out, lse = st.results()
        assert fnpu.check() == fnpu.FNPU_OK
        ref_o, ref_l = _oracle_after_append(batch)
        assert np.abs(out - ref_o).max() <= O_TOL and np.abs(lse - ref_l).max() <= LSE_TOL

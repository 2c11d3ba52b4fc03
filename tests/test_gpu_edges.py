"""Kernels and dispatch rules at the sizes where they can go wrong: tile remainders, the smallest and largest of a range,
the points where one variant hands over to another.  Tolerances are those of parity_util and test_gpu_decode."""
import numpy as np
import pytest
import torch

import oracle
import rkv_inputs as ri
from test_gpu_parity import rkv, run_and_check, small_spec  # noqa: F401  (rkv: the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,beta,T", [("bf16", 1, 0.5), ("bf16", 3, 0.5), ("bf16", 1, 0.9), ("fp8", 2, 0.5)])
@pytest.mark.parametrize("budget,buffer,lens", [(100, 36, [136, 135, 101]), (256, 137, [393, 265, 264]), (17, 8, [25, 18, 17])])
def test_row_block_scoring_of_256_dimensions(rkv, dtype, beta, T, budget, buffer, lens):  # noqa: F811
    """Operand tiles in two 128-column blocks: one row tile and two, n = 128, 127, 385, 257, 256, a cache of one small tile."""
    spec = small_spec("rb256", batch=3, hkv=2, hq=8, budget=budget, buffer=buffer, head_dim=256, dtype=dtype, span=8)
    wl = ri.make_workload(spec, device="cuda", seed=401 + budget, seq_lens=torch.tensor(lens))
    rep, comp = run_and_check(rkv, wl, beta=beta, T=T)
    assert rep.ok(), rep.errors
    assert rep.compressed_heads == 2 * sum(L > budget for L in lens)
    comp.check_status()


@pytest.mark.parametrize("dtype,beta,T", [("bf16", 1, 0.5), ("bf16", 3, 0.5), ("bf16", 1, 0.95), ("fp8", 1, 0.5)])
@pytest.mark.parametrize("budget,buffer,lens", [(100, 36, [136, 135, 101]), (256, 137, [393, 265, 264]), (17, 8, [25, 18, 17]),
                                                (1500, 164, [1664, 1545, 1544])])
def test_two_pass_scoring_of_64_dimensions(rkv, dtype, beta, T, budget, buffer, lens):  # noqa: F811
    """Units of two key tiles: even and odd numbers of tiles, a second tile without a candidate, with one, full; the rounds and
    (T = 0.95: hardly any pair) the symmetric route."""
    spec = small_spec("d64", batch=3, hkv=2, hq=8, budget=budget, buffer=buffer, head_dim=64, dtype=dtype, span=8)
    wl = ri.make_workload(spec, device="cuda", seed=405 + budget, seq_lens=torch.tensor(lens))
    for b, L in enumerate(lens):
        wl.k_cache.view(torch.int16 if dtype == "bf16" else torch.uint8)[b, :, L:] = 0x7FC0 if dtype == "bf16" else 0x7F      # NaN
    rep, comp = run_and_check(rkv, wl, beta=beta, T=T)
    assert rep.ok(), rep.errors
    assert rep.compressed_heads == 2 * sum(L > budget for L in lens)
    comp.check_status()


@pytest.mark.parametrize("head_dim,hq,alpha", [(64, 2, 8), (128, 8, 8), (128, 18, 8), (256, 6, 5)])
@pytest.mark.parametrize("budget,buffer,lens", [(40, 32, [72, 71, 41]), (110, 90, [200, 137, 136])])
def test_cuda_core_scoring_tiles(rkv, head_dim, hq, alpha, budget, buffer, lens):  # noqa: F811
    """64-row blocks and 64- (d = 256: 32-) key steps: n = 64, 63, 33, 192, 129, 128; one and two passes over the query rows
    (72 rows: more than a block of 64)."""
    spec = small_spec("simt", batch=3, hkv=2, hq=hq, budget=budget, buffer=buffer, alpha=alpha, head_dim=head_dim, dtype="f32", span=8)
    wl = ri.make_workload(spec, device="cuda", seed=411 + hq, seq_lens=torch.tensor(lens))
    for b, L in enumerate(lens):
        wl.k_cache[b, :, L:] = float("nan")
    rep, comp = run_and_check(rkv, wl, beta=2)
    assert rep.ok(), rep.errors
    comp.check_status()


@pytest.mark.parametrize("batch,hkv", [(74, 8), (75, 8), (593, 1)])
def test_lists_of_many_heads(rkv, batch, hkv):  # noqa: F811
    """592, 600 and 593 heads (four per SM on 148): above that a warp lists a head alone.  Two key tiles, a last block of the listing
    that is not full, sequences without anything below their last tile."""
    spec = small_spec("lists", batch=batch, hkv=hkv, hq=hkv, budget=150, buffer=42, span=4, copy_frac=0.2)
    lens = [(192, 191, 151, 150)[b % 4] for b in range(batch)]
    wl = ri.make_workload(spec, device="cuda", seed=408 + batch, seq_lens=torch.tensor(lens))
    rep, comp = run_and_check(rkv, wl)
    assert rep.ok(), rep.errors
    comp.check_status()


@pytest.mark.parametrize("batch,hkv,alpha,pool_w,beta", [(38, 8, 8, 4, 1), (37, 8, 8, 4, 3), (300, 1, 5, 2, 1)])
def test_many_small_heads(rkv, batch, hkv, alpha, pool_w, beta):  # noqa: F811
    """304, 296 and 300 heads: the selection's blocks halve above two heads per SM (296 on 148 SMs).  n = 128, 127, 93, lists that
    end inside a warp's piece."""
    spec = small_spec("many", batch=batch, hkv=hkv, hq=2 * hkv, budget=100, buffer=36, alpha=alpha, span=4)
    lens = [(136, 135, 101, 100)[b % 4] for b in range(batch)]
    wl = ri.make_workload(spec, device="cuda", seed=407 + batch, seq_lens=torch.tensor(lens))
    rep, comp = run_and_check(rkv, wl, beta=beta, W=pool_w)
    assert rep.ok(), rep.errors
    comp.check_status()


@pytest.mark.parametrize("batch,hkv,hq,cap", [(1, 1, 4, 128), (1, 1, 4, 8192), (2, 1, 8, 2176), (1, 2, 2, 1920), (1, 2, 2, 1921),
                                              (40, 8, 16, 640)])
def test_decode_attention_splits(rkv, batch, hkv, hq, cap):  # noqa: F811
    """One block per head up to the largest cluster (16 blocks), more key tiles than one block holds (15), many heads with a
    single split; lengths that leave the last blocks of a cluster without a row."""
    spec = ri.CacheSpec("split", 1, batch, hkv, hq, 128, cap - 64, 64, 8, 0.1, "bf16", 16, 0.3, 0.05, 4, 8.0)
    lens = [(cap, cap - 1, 1, cap // 2, 129)[b % 5] if b else cap for b in range(batch)]
    if batch == 1:
        lens = [max(1, cap - 130)]
    wl = ri.make_workload(spec, device="cuda", seed=421, seq_lens=torch.tensor(lens))
    for b, L in enumerate(lens):
        wl.k_cache[b, :, L:] = float("nan")
        wl.v_cache[b, :, L:] = float("nan")
    g = torch.Generator(device="cuda").manual_seed(7)
    q_new = torch.randn(batch, hq, 128, generator=g, device="cuda").to(torch.bfloat16)
    comp = rkv.Compressor(batch, hkv, hq, spec.budget, spec.buffer, spec.alpha, 0.1)
    out = torch.full((batch, hq, 128), 7.0, device="cuda")
    for _ in range(2):                              # back to back: the second starts while the first is still running
        assert rkv.rkv_decode_attention(comp.desc, wl.k_cache, wl.v_cache, q_new, wl.seq_lens, out, spec.budget, spec.buffer) == 0
    torch.cuda.synchronize()
    comp.check_status()
    K, V = (torch.nan_to_num(t.float(), nan=0.0).cpu().numpy() for t in (wl.k_cache, wl.v_cache))
    ref = oracle.oracle_decode_attention(K, V, q_new.float().cpu().numpy(), np.array(lens, dtype=np.int32))
    got = out.cpu().numpy().astype(np.float64)
    scale = np.maximum(np.abs(ref).max(axis=-1, keepdims=True), 1e-30)
    assert (np.abs(got - ref) <= 1e-3 * scale + 1e-7).all(), float((np.abs(got - ref) / scale).max())


@pytest.mark.parametrize("dtype,head_dim", [("fp8", 128), ("bf16", 64), ("bf16", 128)])
@pytest.mark.parametrize("heads,cap", [(296, 2176), (297, 2176), (200, 4224)])
def test_decode_attention_splits_as_blocks(rkv, dtype, head_dim, heads, cap):  # noqa: F811
    """Two waves of blocks on 148 SMs (two splits of 296 heads: clusters) and more (8-bit caches and 64 dimensions: blocks of their
    own, partial results in the workspace, here full of NaN): lengths that leave the last splits without a row, none at all."""
    group = 4
    g = torch.Generator(device="cuda").manual_seed(heads)
    k, v = (torch.randn(heads, 1, cap, head_dim, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    dt = torch.float8_e4m3fn if dtype == "fp8" else torch.bfloat16
    k, v = k.to(dt), v.to(dt)
    q_new = torch.randn(heads, group, head_dim, generator=g, device="cuda").to(torch.bfloat16)
    lens = torch.tensor([(cap, cap - 1, 1, 130, 0, cap // 2)[b % 6] for b in range(heads)], dtype=torch.int32)
    for b, L in enumerate(lens.tolist()):
        for t in (k, v):
            t.view(torch.uint8 if dtype == "fp8" else torch.int16)[b, :, L:] = 0x7F if dtype == "fp8" else 0x7FC0
    comp = rkv.Compressor(heads, 1, group, cap - 64, 64, 8, 0.1, dtype=dt, head_dim=head_dim)
    comp.workspace.fill_(0xFF)
    out = torch.full((heads, group, head_dim), 7.0, device="cuda")
    for _ in range(2):
        assert rkv.rkv_decode_attention(comp.desc, k, v, q_new, lens.cuda(), out, cap - 64, 64) == 0
    torch.cuda.synchronize()
    comp.check_status()
    rows = [0, 1, 2, 3, 4, 5, heads - 6, heads - 5, heads - 4, heads - 3, heads - 2, heads - 1]
    K, V = (torch.nan_to_num(t.view(torch.uint8)[rows].view(t.dtype).float() if dtype == "fp8" else t[rows].float(), nan=0.0).cpu().numpy()
            for t in (k, v))
    ref = oracle.oracle_decode_attention(K, V, q_new[rows].float().cpu().numpy(), lens[rows].numpy())
    got = out[rows].cpu().numpy().astype(np.float64)
    assert np.isfinite(out.cpu().numpy()).all()
    scale = np.maximum(np.abs(ref).max(axis=-1, keepdims=True), 1e-30)
    assert (np.abs(got - ref) <= 1e-3 * scale + 1e-7).all(), float((np.abs(got - ref) / scale).max())


@pytest.mark.parametrize("cap,nan_rows", [(1920, (0, 128)), (1920, (0, 1920)), (1920, (1152, 1280)), (1280, (5, 6))])
def test_decode_attention_over_nan_keys(rkv, cap, nan_rows):  # noqa: F811
    """Keys of NaN give the output row that they give when one block holds the head (zeros: no sum of weights), also when they are
    all that a block of the cluster holds; a sequence without any is not touched by them."""
    batch, hkv, hq = 2, 1, 4
    g = torch.Generator(device="cuda").manual_seed(9)
    k, v = (torch.randn(batch, hkv, cap, 128, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    q_new = torch.randn(batch, hq, 128, generator=g, device="cuda").to(torch.bfloat16)
    k[0, :, nan_rows[0]:nan_rows[1]] = float("nan")
    comp = rkv.Compressor(batch, hkv, hq, cap - 64, 64, 8, 0.1)
    lens = torch.full((batch,), cap, dtype=torch.int32, device="cuda")
    out = torch.full((batch, hq, 128), 7.0, device="cuda")
    assert rkv.rkv_decode_attention(comp.desc, k, v, q_new, lens, out, cap - 64, 64) == 0
    torch.cuda.synchronize()
    comp.check_status()
    assert not out[0].any()
    ref = oracle.oracle_decode_attention(k[1:].float().cpu().numpy(), v[1:].float().cpu().numpy(), q_new[1:].float().cpu().numpy(),
                                         np.array([cap], dtype=np.int32))
    got = out[1:].cpu().numpy().astype(np.float64)
    assert (np.abs(got - ref) <= 1e-3 * np.abs(ref).max(axis=-1, keepdims=True) + 1e-7).all()


@pytest.mark.parametrize("hkv,head_dim,dtype", [(1, 64, torch.bfloat16), (32, 128, torch.float32), (512, 128, torch.bfloat16),
                                                (513, 128, torch.bfloat16)])
def test_append_rows_of_one_block(rkv, hkv, head_dim, dtype):  # noqa: F811
    """A sequence's new rows are moved by one block: 8 vectors and 1024 (several per thread), up to 8192; by several from there on; appends
    in a row, the last one into a cache that is full by then."""
    batch, budget, buffer = 3, 24, 8
    cap = budget + buffer
    comp = rkv.Compressor(batch, hkv, hkv, budget, buffer, 8, 0.1, dtype=dtype, head_dim=head_dim)
    g = torch.Generator(device="cuda").manual_seed(3)
    k = torch.randn(batch, hkv, cap, head_dim, generator=g, device="cuda").to(dtype)
    v, want_k, want_v = k + 1, k.clone(), k + 1
    lens = torch.tensor([0, cap - 2, cap], dtype=torch.int32, device="cuda")
    length = lens.tolist()
    for step in range(3):
        kn = torch.randn(batch, hkv, head_dim, generator=g, device="cuda").to(dtype)
        vn = kn * 2
        assert rkv.rkv_append(comp.desc, k, v, kn, vn, lens, budget, buffer) == 0
        for b in range(batch):
            if length[b] < cap:
                want_k[b, :, length[b]], want_v[b, :, length[b]] = kn[b], vn[b]
                length[b] += 1
    torch.cuda.synchronize()
    assert lens.tolist() == length == [3, cap, cap]
    assert torch.equal(k, want_k) and torch.equal(v, want_v)
    assert int(comp.status.item()) == 1              # the full cache was reported


@pytest.mark.parametrize("batch", [7, 9, 17])
def test_host_buffers_in_pieces(rkv, batch):  # noqa: F811
    """The host-buffer form cuts larger batches into pieces of whole sequences: one piece (33 MB of caches), uneven ones (42 and 80), two
    calls in a row on the same buffers' copies, ragged lengths, per-sequence budgets."""
    spec = small_spec("pieces", batch=batch, hkv=8, hq=16, budget=1024, buffer=128, span=32)
    lens = [spec.cap - 9 * (b % 5) for b in range(batch)]
    lens[2] = 900
    budgets = torch.tensor([spec.budget - 13 * (b % 3) for b in range(batch)])
    wl = ri.make_workload(spec, device="cuda", seed=431, seq_lens=torch.tensor(lens))
    ch = rkv.Compressor(batch, 8, 16, spec.budget, spec.buffer, 8, 0.1, host_staging=True, budgets=budgets)
    sets = [[t.cpu().pin_memory() for t in (wl.k_cache, wl.v_cache, wl.q_window, wl.seq_lens)] for _ in range(2)]
    got = []
    for hk, hv, hq, hs in sets:                     # (nothing between the calls waits for the GPU)
        got.append((hk, hv, hs, torch.empty(batch, 8, spec.budget, dtype=torch.int32, pin_memory=True)))
    for (hk, hv, hq, hs), (_, _, _, hidx) in zip(sets, got):
        ch.compress_host(hk, hv, hq, hs, hidx)
    cd = rkv.Compressor(batch, 8, 16, spec.budget, spec.buffer, 8, 0.1, budgets=budgets)
    idx = cd.compress(wl.k_cache, wl.v_cache, wl.q_window, wl.seq_lens)
    torch.cuda.synchronize()
    ch.check_status()
    for hk, hv, hs, hidx in got:
        assert torch.equal(hidx, idx.cpu()) and torch.equal(hs, wl.seq_lens.cpu())
        for b in range(batch):
            n = int(hs[b])
            assert torch.equal(hk[b, :, :n].view(torch.int16), wl.k_cache[b, :, :n].cpu().view(torch.int16))
            assert torch.equal(hv[b, :, :n].view(torch.int16), wl.v_cache[b, :, :n].cpu().view(torch.int16))


def test_host_buffers_on_independent_streams(rkv):  # noqa: F811
    """A call in pieces on one stream does not wait for the copies of a call whose own stream is busy with something else."""
    batch = 9                                            # 42 MB of caches: two pieces
    spec = small_spec("streams", batch=batch, hkv=8, hq=16, budget=1024, buffer=128, span=32)
    wl = ri.make_workload(spec, device="cuda", seed=433)
    sets = []
    for _ in range(3):
        comp = rkv.Compressor(batch, 8, 16, spec.budget, spec.buffer, 8, 0.1, host_staging=True)
        sets.append((comp, [t.cpu().pin_memory() for t in (wl.k_cache, wl.v_cache, wl.q_window, wl.seq_lens)],
                     torch.empty(batch, 8, spec.budget, dtype=torch.int32).pin_memory()))
    torch.cuda.synchronize()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    for (comp, host, hidx), stream in zip(sets, (a, a, b)):
        with torch.cuda.stream(stream):
            if comp is sets[1][0]:
                torch.cuda._sleep(1_000_000_000)         # about half a second of the first stream, on which its second call waits
            comp.compress_host(*host, hidx, stream)
    b.synchronize()
    assert not a.query()
    a.synchronize()
    want = sets[0]
    for comp, host, hidx in sets:
        comp.check_status()
        assert torch.equal(hidx, want[2]) and torch.equal(host[3], want[1][3])
        for x, y in zip(host[:2], want[1][:2]):
            assert torch.equal(x[:, :, :spec.budget].view(torch.int16), y[:, :, :spec.budget].view(torch.int16))


@pytest.mark.parametrize("head_dim,dtype,batch", [(64, "fp8", 19), (64, "bf16", 19), (128, "bf16", 19), (256, "bf16", 19), (256, "f32", 19),
                                                  (64, "fp8", 28), (64, "bf16", 28), (128, "bf16", 28), (128, "bf16", 27), (256, "bf16", 18),
                                                  (128, "bf16", 511), (128, "bf16", 512)])
@pytest.mark.parametrize("pattern", ["runs", "last_k", "sparse", "identity"])
def test_compaction_by_bulk_copies(rkv, head_dim, dtype, batch, pattern):  # noqa: F811
    """The gather stage alone on hand-made ascending lists, every row width, eight streams per sequence on both sides of the lines between its
    kernels (222 streams on 148 SMs, 148 for rows of 512 bytes and more, 4096 for rows of 256); runs that cross chunks,
    single rows, a long shift, a list in place already, a budget that is not a whole number of chunks; ragged lengths."""
    hkv, budget, buffer, alpha = 4, 333, 83, 8
    spec = small_spec("bulk", batch=batch, hkv=hkv, hq=hkv, budget=budget, buffer=buffer, head_dim=head_dim, dtype=dtype)
    cap = spec.cap
    lens = torch.tensor([budget - 5 if b % 7 == 3 else cap - b % 5 for b in range(batch)])
    wl = ri.make_workload(spec, device="cuda", seed=441, seq_lens=lens)
    comp = rkv.Compressor(batch, hkv, hkv, budget, buffer, alpha, 0.1, dtype=spec.torch_dtype, head_dim=head_dim)
    comp.compress(wl.k_cache, wl.v_cache, wl.q_window, wl.seq_lens, stages=rkv.RKV_STAGE_PREP)       # records lengths
    g = torch.Generator().manual_seed(5)
    idx = torch.empty(batch, hkv, budget, dtype=torch.int32)
    for b in range(batch):
        L = int(lens[b])
        for h in range(hkv):
            if pattern == "identity" or L <= budget:
                row = torch.arange(budget)
            elif pattern == "last_k":
                row = torch.arange(L - budget, L)
            elif pattern == "sparse":
                row = torch.randperm(L, generator=g)[:budget].sort().values
            else:                                    # what is dropped comes in spans
                keep = torch.ones(L, dtype=torch.bool)
                drop = L - budget
                start = int(torch.randint(0, L - drop, (1,), generator=g))
                keep[start:start + drop] = False
                row = keep.nonzero().flatten()
            idx[b, h] = row.int()
    comp.out_idx.copy_(idx)
    u8 = lambda t: t.view(torch.uint8)  # noqa: E731
    k0, v0 = u8(wl.k_cache).clone(), u8(wl.v_cache).clone()
    comp.compress(wl.k_cache, wl.v_cache, wl.q_window, wl.seq_lens, stages=rkv.RKV_STAGE_GATHER)
    torch.cuda.synchronize()
    comp.check_status()
    take = idx.long().cuda()[..., None].expand(-1, -1, -1, k0.shape[-1])
    assert torch.equal(u8(wl.k_cache)[:, :, :budget], k0.gather(2, take))
    assert torch.equal(u8(wl.v_cache)[:, :, :budget], v0.gather(2, take))
    assert wl.seq_lens.tolist() == [min(int(x), budget) for x in lens]


@pytest.mark.parametrize("dtype,head_dim,tile", [("f32", 128, 0), ("f32", 64, 2), ("bf16", 256, 0), ("bf16", 256, 2)])
def test_norms_of_a_tile_given_up_abort_the_call(rkv, dtype, head_dim, tile):  # noqa: F811
    """What a prep block that gave up leaves behind (-1 as the first norm of a tile), put there by hand between the stages: the
    scoring kernel records the abort."""
    spec = small_spec("mark", batch=3, hkv=2, hq=4, budget=300, buffer=84, head_dim=head_dim, dtype=dtype, span=8)
    wl = ri.make_workload(spec, device="cuda", seed=453)
    k0, s0 = wl.k_cache.clone(), wl.seq_lens.clone()
    comp = rkv.Compressor(3, 2, 4, spec.budget, spec.buffer, spec.alpha, 0.1, dtype=spec.torch_dtype, head_dim=head_dim)
    comp.compress(wl.k_cache, wl.v_cache, wl.q_window, wl.seq_lens, stages=rkv.RKV_STAGE_PREP)
    norms = comp.workspace[:6 * 384 * 4].view(torch.float32).view(6, 384)       # no copy of the keys: they come first
    assert bool((norms[:, :300] > 0).all())
    norms[4, 128 * tile] = -1.0
    rest = rkv.RKV_STAGE_SCORES | rkv.RKV_STAGE_SELECT | rkv.RKV_STAGE_GATHER
    comp.compress(wl.k_cache, wl.v_cache, wl.q_window, wl.seq_lens, stages=rest)
    torch.cuda.synchronize()
    assert int(comp.status.item()) == 5
    assert torch.equal(wl.k_cache, k0) and torch.equal(wl.seq_lens, s0) and bool((comp.out_idx == -1).all())


@pytest.mark.parametrize("budget,buffer", [(600, 100), (1900, 100)])
def test_logits_of_minus_infinity(rkv, budget, buffer):  # noqa: F811
    """Products that overflow to -inf weigh nothing in the softmax of Eq. 3, also where they are all that a lane sees (the lanes of the
    row statistics take four of every 128 tokens): single-kernel and three-kernel selection."""
    spec = small_spec("inf", batch=1, hkv=1, hq=1, budget=budget, buffer=buffer, span=8)
    wl = ri.make_workload(spec, device="cuda", seed=461)
    pos = torch.arange(spec.cap, device="cuda")
    low = (pos % 128 >= 40) & (pos % 128 < 48)
    wl.q_window.fill_(1e30)
    wl.k_cache[:] = torch.where(low[:, None], -1e10, 0.0).to(torch.bfloat16)
    wl.k_cache[0, 0, :, 0] += torch.where(low, 0.0, (pos % 7).float() * 1e-30).to(torch.bfloat16)
    rep, comp = run_and_check(rkv, wl)
    assert rep.ok(), rep.errors
    comp.check_status()


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("beta,T", [(4, 0.5), (5, 0.5), (8, 0.3), (40, 0.2)])
def test_first_pass_partners_of_a_chunk(rkv, head_dim, beta, T):  # noqa: F811
    """Up to four partners of a chunk are taken out one by one, more in one sum: copies in abundance, counts on both sides within a
    warp, partners that run out in the middle of a chunk."""
    spec = small_spec("chunk", batch=2, hkv=2, hq=4, budget=150, buffer=100, head_dim=head_dim, span=2, copy_frac=0.7)
    wl = ri.make_workload(spec, device="cuda", seed=463 + beta, seq_lens=torch.tensor([250, 201]))
    rep, comp = run_and_check(rkv, wl, beta=beta, T=T)
    assert rep.ok(), rep.errors
    comp.check_status()


SECOND_CONTEXT = """
import ctypes, sys
import torch
import paper_2505_24133_b200 as rkv
cu = ctypes.CDLL("libcuda.so.1")
P = ctypes.c_void_p

def call():
    d = rkv.rkv_desc_default()
    d.batch, d.n_kv_heads, d.n_q_heads = 2, 4, 8
    need, cap = rkv.rkv_workspace_bytes(d, 300, 84, 8), 384

    def device(nbytes, fill=0x3f):
        p = P()
        assert cu.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(nbytes)) == 0 and cu.cuMemsetD8_v2(p, ctypes.c_ubyte(fill), ctypes.c_size_t(nbytes)) == 0
        return p.value
    d.workspace, d.workspace_bytes = device(need, 0), need
    k, v, q, idx = device(8 * cap * 256), device(8 * cap * 256), device(2 * 8 * 8 * 256), device(8 * 300 * 4)
    lens = device(8, 0)
    assert cu.cuMemsetD32_v2(P(lens), ctypes.c_uint(cap), ctypes.c_size_t(2)) == 0
    out = device(2 * 8 * 128 * 4)
    rc = rkv.rkv_compress_stages(d, k, v, q, lens, 300, 84, 8, 0.1, idx, 0)
    rc2 = rkv.rkv_decode_attention(d, k, v, q, lens, out, 300, 84, 0)
    assert cu.cuCtxSynchronize() == 0
    got = (ctypes.c_int * 2)()
    assert cu.cuMemcpyDtoH_v2(got, P(lens), ctypes.c_size_t(8)) == 0
    return rc, rc2, list(got)

torch.zeros(1, device="cuda")                       # the primary context
first = call()
ctx, dev = P(), ctypes.c_int()
assert cu.cuDeviceGet(ctypes.byref(dev), 0) == 0 and cu.cuCtxCreate_v2(ctypes.byref(ctx), 0, dev) == 0
second = call()
print(first, second)
sys.exit(0 if first == second == (0, 0, [300, 300]) else 1)
"""


def test_calls_in_a_second_context_of_the_device(rkv):  # noqa: F811
    """Function attributes belong to a context: kernels prepared in one are prepared again in another."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", SECOND_CONTEXT], cwd=root, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, PYTHONPATH=root))
    assert r.returncode == 0, r.stdout + r.stderr[-2000:]

"""The two-pass scoring route at the sizes where its kernels can go wrong.  Tolerances are those of parity_util."""
import pytest
import torch

import rkv_inputs as ri
from parity_util import check_batch, pick
from test_gpu_parity import DEFAULTS, rkv, run_and_check, small_spec  # noqa: F401  (rkv: the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("head_dim,dtype", [(64, "bf16"), (128, "bf16"), (128, "fp8")])
@pytest.mark.parametrize("hq,alpha,mean", [(1, 8, False), (7, 8, False), (14, 8, False), (14, 8, True), (9, 12, False), (3, 5, True)])
def test_logits_of_the_prep_stage(rkv, head_dim, dtype, hq, alpha, mean):  # noqa: F811
    """Query blocks of 16 to 112 rows (64 dimensions: four groups' accumulators up to 48 rows, three at 64, two above), other window lengths than
    eight, the mean over the group; units without a candidate, heads that change inside a block's range (24 heads of four tiles)."""
    lens = [(512, 385, 384, 257, 300, 400)[b % 6] for b in range(12)]
    spec = small_spec("logits", batch=12, hkv=2, hq=2 * hq, budget=300, buffer=212, alpha=alpha, head_dim=head_dim, dtype=dtype, span=8)
    wl = ri.make_workload(spec, device="cuda", seed=541 + hq, seq_lens=torch.tensor(lens))
    for b, L in enumerate(lens):
        wl.k_cache.view(torch.int16 if dtype == "bf16" else torch.uint8)[b, :, L:] = 0x7FC0 if dtype == "bf16" else 0x7F      # NaN
    rep, comp = run_and_check(rkv, wl, flags=rkv.RKV_FLAG_GQA_MEAN_POOL if mean else 0)
    assert rep.ok(), rep.errors
    assert rep.compressed_heads == 2 * sum(L > 300 for L in lens)
    comp.check_status()


@pytest.mark.parametrize("hq", [16, 64, 112])
@pytest.mark.parametrize("head_dim,dtype", [(64, "bf16"), (128, "bf16"), (128, "fp8")])
def test_logits_where_blocks_take_many_units(rkv, head_dim, dtype, hq):  # noqa: F811
    """1600 heads of two tiles: every block's range runs over many heads, so query blocks and ring stages are used over and over; with 16,
    64 and 112 query rows the ring has more stages than there are groups, and as many."""
    spec = small_spec("range", batch=200, hkv=8, hq=hq, budget=150, buffer=42, head_dim=head_dim, dtype=dtype, span=8)
    lens = [(192, 191, 151, 150)[b % 4] for b in range(200)]
    wl = ri.make_workload(spec, device="cuda", seed=551, seq_lens=torch.tensor(lens))
    rep, comp = run_and_check(rkv, wl, check_rows=[0, 1, 2, 98, 99, 100, 101, 197, 198])
    assert rep.ok(), rep.errors
    comp.check_status()


@pytest.mark.parametrize("hq", [8, 32, 112])
@pytest.mark.parametrize("head_dim,dtype", [(64, "bf16"), (128, "bf16"), (128, "fp8")])
@pytest.mark.parametrize("budget,buffer", [(60, 36), (200, 184), (420, 92)])
def test_logits_of_short_heads(rkv, head_dim, dtype, hq, budget, buffer):  # noqa: F811
    """2400 heads of one, three and four tiles (64 dimensions: one or two units): as many heads' queries are under way as the ring of units
    reaches over; sequences that are not compressed, whose queries nobody asks for, lie between the others."""
    cap = budget + buffer
    some = [cap, budget + 1, budget, cap - 1, 3, cap, 0, budget + buffer // 2]
    lens = [some[b % 7 if b < 280 else 2] for b in range(300)]
    spec = small_spec("short", batch=300, hkv=8, hq=hq, budget=budget, buffer=buffer, head_dim=head_dim, dtype=dtype, span=8)
    wl = ri.make_workload(spec, device="cuda", seed=555 + budget, seq_lens=torch.tensor(lens))
    rep, comp = run_and_check(rkv, wl, check_rows=[0, 1, 2, 3, 5, 100, 101, 150, 199, 278, 279, 299])
    assert rep.ok(), rep.errors
    comp.check_status()


@pytest.mark.parametrize("beta,T", [(1, 0.5), (1, 0.95), (3, 0.5), (1, 1.0)])
@pytest.mark.parametrize("budget,buffer,lens", [(100, 28, [128, 127, 101]), (100, 36, [136, 135, 101]), (1500, 164, [1664, 1545, 1501])])
def test_codes_scored_as_they_are_stored(rkv, beta, T, budget, buffer, lens):  # noqa: F811
    """E4M3 codes of 128 dimensions: capacities of a whole number of tiles and others, one tile, both rounds, the symmetric route (T =
    0.95, 13 tiles), several partners, the rule off; the values the codes stand for span eight octaves."""
    spec = small_spec("codes", batch=3, hkv=2, hq=8, budget=budget, buffer=buffer, dtype="fp8", span=8)
    wl = ri.make_workload(spec, device="cuda", seed=561 + budget, seq_lens=torch.tensor(lens))
    scale = torch.exp2(torch.randint(-4, 4, (spec.cap, 1), generator=torch.Generator().manual_seed(5)).float()).cuda()
    wl.k_cache.copy_((wl.k_cache.float() * scale).clamp(-448, 448).to(torch.float8_e4m3fn))
    for b, L in enumerate(lens):
        wl.k_cache.view(torch.uint8)[b, :, L:] = 0x7F      # NaN
    rep, comp = run_and_check(rkv, wl, beta=beta, T=T)
    assert rep.ok(), rep.errors
    assert rep.compressed_heads == 2 * sum(L > budget for L in lens)
    comp.check_status()


@pytest.mark.parametrize("budget,buffer", [(500, 140), (500, 150)])
def test_codes_by_either_route(rkv, budget, buffer):  # noqa: F811
    """The codes as they are against their widened copy (row-block kernel), both kinds of capacity: the same lists."""
    spec = small_spec("routes8", batch=2, hkv=2, hq=8, budget=budget, buffer=buffer, dtype="fp8", span=8)
    wl = ri.make_workload(spec, device="cuda", seed=571, seq_lens=torch.tensor([640, 601]))
    got = []
    for flags in (0, rkv.RKV_FLAG_ROWBLOCK_SCORES):
        k, v, lens = wl.k_cache.clone(), wl.v_cache.clone(), wl.seq_lens.clone()
        comp = rkv.Compressor(2, 2, 8, budget, buffer, 8, 0.1, dtype=torch.float8_e4m3fn, flags=flags)
        idx = comp.compress(k, v, wl.q_window, lens)
        torch.cuda.synchronize()
        comp.check_status()
        got.append(idx.clone())
    assert torch.equal(got[0], got[1])


@pytest.mark.parametrize("route", ["ROWBLOCK_SCORES", "SIMT_SCORES", "stages"])
@pytest.mark.parametrize("paged", [False, True])
def test_copy_where_blocks_take_many_units(rkv, route, paged):  # noqa: F811
    """The widened copy of 1600 heads of two whole tiles, which the prep kernel writes (also where prep and scores are calls of their own):
    every group of warps takes several units, so operand tiles are written again behind their own stores; lengths inside
    a tile, sequences that are not compressed, pages of other owners full of NaN."""
    from parity_util import from_paged, random_block_table, to_paged
    budget, buffer, B = 180, 76, 200
    lens = [(256, 255, 181, 180, 129)[b % 5] for b in range(B)]
    spec = small_spec("copies", batch=B, hkv=8, hq=8, budget=budget, buffer=buffer, dtype="fp8", span=8)
    wl = ri.make_workload(spec, device="cuda", seed=577, seq_lens=torch.tensor(lens))
    k0, v0, q0, s0 = wl.k_cache.clone(), wl.v_cache.clone(), wl.q_window.clone(), wl.seq_lens.clone()
    k, v, more = wl.k_cache, wl.v_cache, {}
    if paged:
        pool_pages = B * 8 * 2 + 11
        table = random_block_table(B, 8, 2, pool_pages, seed=15)
        k, v = (to_paged(t.view(torch.uint8), pool_pages, table, fill=0x7F).view(t.dtype) for t in (k, v))
        more = dict(block_table=table, pool_pages=pool_pages)
    comp = rkv.Compressor(B, 8, 8, budget, buffer, spec.alpha, spec.lam, dtype=spec.torch_dtype, dump_scores=True,
                          flags=0 if route == "stages" else getattr(rkv, "RKV_FLAG_" + route), **more)
    for st in (rkv.RKV_STAGE_PREP, rkv.RKV_STAGE_ALL & ~rkv.RKV_STAGE_PREP) if route == "stages" else (rkv.RKV_STAGE_ALL,):
        idx = comp.compress(k, v, wl.q_window, wl.seq_lens, stages=st)
    torch.cuda.synchronize()
    comp.check_status()
    if paged:
        k, v = (from_paged(t.view(torch.uint8), table).view(t.dtype) for t in (k, v))
    sel = torch.tensor([0, 1, 2, 3, 4, 70, 71, 72, 140, 141, 197, 198, 199], device="cuda")
    rep = check_batch(*(pick(t, sel) for t in (k0, v0)), q0[sel], s0[sel], budget=budget, alpha=spec.alpha, lam=spec.lam, gpu_idx=idx[sel],
                      gpu_k=pick(k, sel), gpu_v=pick(v, sel), gpu_seq=wl.seq_lens[sel], gpu_scores=comp.scores[:, sel], **DEFAULTS)
    assert rep.ok(), rep.errors
    assert rep.compressed_heads == 8 * sum(lens[i] > budget for i in sel.tolist())


@pytest.mark.parametrize("size", [0.0, 1e-3, 1.0, 400.0])
def test_key_sums_of_codes(rkv, size):  # noqa: F811
    """The head's key sum travels as codes in parts of falling weight: keys of one value, of the smallest and of the largest codes, none."""
    spec = small_spec("sums", batch=1, hkv=1, hq=1, budget=300, buffer=100, dtype="fp8", span=1, copy_frac=0.0)
    wl = ri.make_workload(spec, device="cuda", seed=581)
    k = wl.k_cache.float()
    k[..., :64] *= size
    k[..., 64:] *= 0.0 if size == 0.0 else 1.0
    wl.k_cache.copy_(k.clamp(-448, 448).to(torch.float8_e4m3fn))
    rep, comp = run_and_check(rkv, wl)
    assert rep.ok(), rep.errors
    comp.check_status()


@pytest.mark.parametrize("head_dim,dtype", [(64, "bf16"), (128, "bf16"), (128, "fp8")])
@pytest.mark.parametrize("beta,T,span", [(1, 0.95, 1), (1, 0.5, 1), (2, 0.5, 16)])
@pytest.mark.parametrize("budget,buffer,batch", [(120, 40, 40), (250, 150, 25), (1300, 100, 13)])
def test_second_pass_items_in_a_row(rkv, head_dim, dtype, beta, T, span, budget, buffer, batch):  # noqa: F811
    """Items of one and of two row tiles behind one another on every SM (resident tiles are taken in turn, three or four of them): T =
    0.95 lists nearly every token (129 to 152 of them, 384 to 392: two items, of two row tiles and of one or two; 1392: six), T = 0.5
    few (one row tile, its key tiles dealt out to both halves)."""
    some = [budget + buffer, budget + buffer - 15, budget + 17, budget + 9]
    lens = [some[b % 4] for b in range(batch)]
    spec = small_spec("items", batch=batch, hkv=8, hq=8, budget=budget, buffer=buffer, head_dim=head_dim, dtype=dtype, span=span, copy_frac=0.5)
    wl = ri.make_workload(spec, device="cuda", seed=501 + budget, seq_lens=torch.tensor(lens))
    for b, L in enumerate(lens):
        wl.k_cache.view(torch.int16 if dtype == "bf16" else torch.uint8)[b, :, L:] = 0x7FC0 if dtype == "bf16" else 0x7F      # NaN
    rows = sorted({0, 1, 2, 3, batch // 2, batch - 2, batch - 1})
    rep, comp = run_and_check(rkv, wl, beta=beta, T=T, flags=rkv.RKV_FLAG_NO_SYMMETRIC, check_rows=rows)
    assert rep.ok(), rep.errors
    comp.check_status()


@pytest.mark.parametrize("dtype,head_dim,hq", [("bf16", 128, 4), ("bf16", 128, 8), ("fp8", 128, 3), ("bf16", 64, 1)])
@pytest.mark.parametrize("heads,cap", [(148, 4224), (296, 2176), (148, 7040)])
def test_decode_attention_in_two_chunks(rkv, dtype, head_dim, hq, heads, cap):  # noqa: F811
    """Blocks of more key tiles than their columns hold the scores of (17 and 28 tiles, two to a head; 17, one): lengths that end in the
    first chunk, at its last row, in the second, at a block's first row; logits far apart between the chunks."""
    import numpy as np
    import oracle
    spec = ri.CacheSpec("chunks", 1, heads, 1, hq, head_dim, cap - 64, 64, 8, 0.1, dtype, 16, 0.3, 0.05, 4, 8.0)
    per = -(-cap // 128) // (1 if heads == 296 else 2) * 128
    some = [cap, cap - 1, 1, 9 * 128, 9 * 128 + 1, 15 * 128, 15 * 128 + 1, 16 * 128 + 5, per, per + 1, 130]
    lens = [min(some[b % len(some)], cap) for b in range(heads)]
    wl = ri.make_workload(spec, device="cuda", seed=611, seq_lens=torch.tensor(lens))
    wl.k_cache[1::3, :, 1500:] = (wl.k_cache[1::3, :, 1500:].float() * 8).clamp(-448, 448).to(wl.k_cache.dtype)
    for b, L in enumerate(lens):
        for t in (wl.k_cache, wl.v_cache):
            t.view(torch.int16 if dtype == "bf16" else torch.uint8)[b, :, L:] = 0x7FC0 if dtype == "bf16" else 0x7F      # NaN
    q_new = torch.randn(heads, hq, head_dim, generator=torch.Generator(device="cuda").manual_seed(7), device="cuda").to(torch.bfloat16)
    comp = rkv.Compressor(heads, 1, hq, spec.budget, spec.buffer, spec.alpha, 0.1, dtype=spec.torch_dtype, head_dim=head_dim)
    out = torch.full((heads, hq, head_dim), 7.0, device="cuda")
    assert rkv.rkv_decode_attention(comp.desc, wl.k_cache, wl.v_cache, q_new, wl.seq_lens, out, spec.budget, spec.buffer) == 0
    torch.cuda.synchronize()
    comp.check_status()
    rows = list(range(0, heads, 13)) + list(range(11))
    K, V = (torch.nan_to_num(t[rows].float(), nan=0.0).cpu().numpy() for t in (wl.k_cache, wl.v_cache))
    ref = oracle.oracle_decode_attention(K, V, q_new[rows].float().cpu().numpy(), np.array([lens[r] for r in rows], dtype=np.int32))
    got = out[rows].cpu().numpy().astype(np.float64)
    scale = np.maximum(np.abs(ref).max(axis=-1, keepdims=True), 1e-30)
    assert (np.abs(got - ref) <= 1e-3 * scale + 1e-7).all(), float((np.abs(got - ref) / scale).max())


@pytest.mark.parametrize("head_dim,dtype,budget,buffer", [(64, "bf16", 300, 100), (128, "bf16", 300, 100), (128, "bf16", 90, 30),
                                                          (128, "fp8", 300, 84), (128, "fp8", 300, 100), (64, "fp8", 300, 84)])
@pytest.mark.parametrize("beta,T", [(1, 0.5), (1, 1.0)])
def test_stages_read_their_inputs_when_they_run(rkv, head_dim, dtype, budget, buffer, beta, T):  # noqa: F811
    """The queries that count are those at the scores; lengths, and 8-bit keys, those at prep: what changes afterwards plays no part."""
    cap = budget + buffer
    lens = [cap, cap - 1, budget + 1, budget]
    spec = small_spec("when", batch=4, hkv=2, hq=8, budget=budget, buffer=buffer, head_dim=head_dim, dtype=dtype, span=8)
    wl = ri.make_workload(spec, device="cuda", seed=591 + budget, seq_lens=torch.tensor(lens))
    k0, v0, q0, s0 = wl.k_cache.clone(), wl.v_cache.clone(), wl.q_window.clone(), wl.seq_lens.clone()
    comp = rkv.Compressor(4, 2, 8, budget, buffer, spec.alpha, 0.1, dtype=spec.torch_dtype, head_dim=head_dim, beta=beta, sim_threshold=T,
                          dump_scores=True)
    args = wl.k_cache, wl.v_cache, wl.q_window, wl.seq_lens
    wl.q_window.normal_(generator=torch.Generator(device="cuda").manual_seed(3)).mul_(4)
    comp.compress(*args, stages=rkv.RKV_STAGE_PREP)
    wl.q_window.copy_(q0)
    wl.seq_lens.copy_(s0.flip(0))
    if dtype == "fp8":
        wl.k_cache.view(torch.uint8).fill_(0x38)
    comp.compress(*args, stages=rkv.RKV_STAGE_SCORES)
    wl.q_window.zero_()
    wl.k_cache.copy_(k0)
    comp.compress(*args, stages=rkv.RKV_STAGE_SELECT)
    wl.seq_lens.copy_(s0)
    idx = comp.compress(*args, stages=rkv.RKV_STAGE_GATHER)
    torch.cuda.synchronize()
    comp.check_status()
    rep = check_batch(k0, v0, q0, s0, budget=budget, alpha=spec.alpha, lam=0.1, gpu_idx=idx, gpu_k=wl.k_cache, gpu_v=wl.v_cache,
                      gpu_seq=wl.seq_lens, gpu_scores=comp.scores, **{**DEFAULTS, "beta": beta, "T": T})
    assert rep.ok(), rep.errors
    assert rep.compressed_heads == 2 * sum(L > budget for L in lens)


@pytest.mark.parametrize("dtype,head_dim,hq", [("bf16", 128, 4), ("fp8", 128, 3), ("bf16", 64, 8)])
@pytest.mark.parametrize("heads,cap", [(8, 1152), (32, 1152), (128, 2176), (296, 2176), (148, 4224), (600, 384)])
@pytest.mark.parametrize("paged", [False, True])
def test_decode_attention_forms(rkv, dtype, head_dim, hq, heads, cap, paged):  # noqa: F811
    """Small grids that fetch before they know the length, large ones, blocks of two chunks: empty sequences, splits without a row, pages
    that a short sequence does not have (-1 in its table).  Weights are carried to 2^-17 each, sums in fp32: that much of the largest output, against 64 bits."""
    import numpy as np
    import oracle
    from parity_util import random_block_table, to_paged
    spec = ri.CacheSpec("forms", 1, heads // 2, 2, 2 * hq, head_dim, cap - 64, 64, 8, 0.1, dtype, 16, 0.3, 0.05, 4, 8.0)
    some = [cap, 0, 1, cap - 1, 128, 129, 0, cap // 2, 300, cap // 2 + 1]
    lens = [min(some[b % len(some)], cap) for b in range(heads // 2)]
    wl = ri.make_workload(spec, device="cuda", seed=621, seq_lens=torch.tensor(lens))
    raw, nan = (torch.int16, 0x7FC0) if dtype == "bf16" else (torch.uint8, 0x7F)
    for b, L in enumerate(lens):
        for t in (wl.k_cache, wl.v_cache):
            t.view(raw)[b, :, L:] = nan
    k, v, more = wl.k_cache, wl.v_cache, {}
    if paged:
        pages = cap // 128
        table = random_block_table(heads // 2, 2, pages, heads * pages + 7, seed=9)
        k, v = (to_paged(t.view(raw), heads * pages + 7, table, fill=nan).view(t.dtype) for t in (k, v))
        for b, L in enumerate(lens):
            table[b, :, -(-L // 128):] = -1
        more = dict(block_table=table, pool_pages=heads * pages + 7)
    q_new = torch.randn(heads // 2, 2 * hq, head_dim, generator=torch.Generator(device="cuda").manual_seed(7), device="cuda").to(torch.bfloat16)
    comp = rkv.Compressor(heads // 2, 2, 2 * hq, spec.budget, spec.buffer, spec.alpha, 0.1, dtype=spec.torch_dtype, head_dim=head_dim, **more)
    out = torch.full((heads // 2, 2 * hq, head_dim), 7.0, device="cuda")
    assert rkv.rkv_decode_attention(comp.desc, k, v, q_new, wl.seq_lens, out, spec.budget, spec.buffer) == 0
    torch.cuda.synchronize()
    comp.check_status()
    rows = list(range(min(10, heads // 2))) + list(range(10, heads // 2, 17))
    K, V = (torch.nan_to_num(t[rows].float(), nan=0.0).cpu().numpy() for t in (wl.k_cache, wl.v_cache))
    ref = oracle.oracle_decode_attention(K, V, q_new[rows].float().cpu().numpy(), np.array([lens[r] for r in rows], dtype=np.int32))
    got = out[rows].cpu().numpy().astype(np.float64)
    err = np.abs(got - ref).max() / np.abs(ref).max()
    assert np.isfinite(got).all() and err <= 2.0 ** -17, err
    assert all(np.all(got[i] == 0.0) for i, r in enumerate(rows) if lens[r] == 0)

"""The two-pass scoring route at the sizes where its kernels can go wrong.  Tolerances are those of parity_util."""
import pytest
import torch

import rkv_inputs as ri
from test_gpu_parity import rkv, run_and_check, small_spec  # noqa: F401  (rkv: the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("head_dim,dtype", [(64, "bf16"), (128, "bf16"), (128, "fp8")])
@pytest.mark.parametrize("hq,alpha,mean", [(1, 8, False), (7, 8, False), (14, 8, False), (14, 8, True), (9, 12, False), (3, 5, True)])
def test_logits_of_the_prep_stage(rkv, head_dim, dtype, hq, alpha, mean):  # noqa: F811
    """Query blocks of 16 to 112 rows (64 dimensions: three groups' accumulators up to 72 rows, two above), other window lengths than
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


@pytest.mark.parametrize("head_dim,dtype", [(64, "bf16"), (128, "bf16"), (128, "fp8")])
def test_logits_where_blocks_take_many_units(rkv, head_dim, dtype):  # noqa: F811
    """1600 heads of two tiles: every block's range runs over many heads, so query blocks and ring stages are used over and over."""
    spec = small_spec("range", batch=200, hkv=8, hq=16, budget=150, buffer=42, head_dim=head_dim, dtype=dtype, span=8)
    lens = [(192, 191, 151, 150)[b % 4] for b in range(200)]
    wl = ri.make_workload(spec, device="cuda", seed=551, seq_lens=torch.tensor(lens))
    rep, comp = run_and_check(rkv, wl, check_rows=[0, 1, 2, 98, 99, 100, 101, 197, 198])
    assert rep.ok(), rep.errors
    comp.check_status()

"""The fp32 attention kernel at the edges of its work split, against the fp64 oracle (GPU only): rows per
lane 1, 2, 4, 6, 8 and their remainders, one to four row groups, contexts on and next to page, warp (128
tokens) and chunk ends.  Tolerance 1e-4 absolute, as everywhere for fp32: sums of up to 2^13 products of
N(0, 1) values in 32 bits, outputs of order 1."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_2601_11652_gb300 import binding as wb  # noqa: E402
from paper_2601_11652_gb300 import workload as wl  # noqa: E402
from paper_2601_11652_gb300.device_batch import DeviceBatch  # noqa: E402


def _check(b):
    db = DeviceBatch.from_host(b)
    db.attention()
    torch.cuda.synchronize()
    assert db.device_status() == (0, -1)
    err = np.max(np.abs(db.results()["out"] - oracle.attention(b)))
    assert err <= 1e-4, err


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("k, Hq, Hkv", [(0, 4, 4), (4, 4, 4), (1, 8, 2), (3, 32, 8), (5, 8, 2), (7, 8, 2), (8, 32, 8),
                                        (12, 28, 4), (23, 8, 2), (15, 16, 2)])
def test_rows_and_contexts(D, k, Hq, Hkv):
    ctx = [0, 1, 15 - min(k, 15), 16, 126, 128, 250, 1000]
    _check(wl.make_batch_from_lengths("f32", draft_lens=[k] * len(ctx), context_lens=ctx, Hq=Hq, Hkv=Hkv, D=D, V=64,
                                      dtype="f32", sigma=0.5, key=(200 + k, D), shuffle_blocks=True))


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("B, ctx", [(1, 9000), (3, 2500)])
def test_chunks(D, B, ctx):
    """Few pairs: sequences cut into chunks whose partials are merged (over 32 of them at B = 1)."""
    _check(wl.make_batch_from_lengths("f32c", draft_lens=[8] * B, context_lens=[ctx + i for i in range(B)], Hq=4, Hkv=1,
                                      D=D, V=64, dtype="f32", sigma=0.5, key=(230, D)))


def test_step_beside_the_acceptance():
    """In a step the attention may be given part of the SMs."""
    b = wl.make_small_batch(61, B=24, Hq=8, Hkv=2, D=128, V=40000, dtype="f32", k_range=(0, 8), ctx_range=(0, 900))
    db = DeviceBatch.from_host(b)
    db.step()
    torch.cuda.synchronize()
    assert db.device_status() == (0, -1)
    got, ref = db.results(), oracle.accept(b)
    assert np.max(np.abs(got["out"] - oracle.attention(b))) <= 1e-4
    near = (ref["accept_margin"] < 1e-6) | (ref["sample_margin"] < 1e-9)
    assert np.all(near | ((got["accepted_len"] == ref["accepted_len"]) & (got["next_token"] == ref["next_token"])))


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("B, ctx", [(40, 700), (1, 9000)])  # whole sequences, and chunks whose partials are merged
def test_keys_of_minus_infinity(D, B, ctx):
    """Keys whose scores are -inf have weight zero: the first page of every warp, a whole chunk, single keys."""
    b = wl.make_batch_from_lengths("inf", draft_lens=[5] * B, context_lens=[ctx + i for i in range(B)], Hq=8, Hkv=4, D=D, V=64,
                                   dtype="f32", sigma=0.5, key=(240, D, B), shuffle_blocks=True)
    b.q[:, :, 0] = np.abs(b.q[:, :, 0]) + np.float32(0.1)
    for r in range(B):
        n = int(b.context_lens[r]) + 6
        for t in [*range(min(640, n // 2)), n // 2 + 1, n - 20]:
            b.k_cache[b.block_tables[r, t // 16], :, t % 16, 0] = -np.inf
    _check(b)


def test_group_times_context_past_31_bits():
    """128 query heads on one KV head and over 2^24 tokens of context: the product of the two does not fit 32
    bits.  The first 4096 keys carry half of every row's weight and a V of their own."""
    heads, D, first, rest = 128, 64, 256, 1 << 20  # pages: `first` times block 0, then the blocks 1 .. 63 in turn
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    kc = torch.randn((64, 1, 16, D), generator=gen, device="cuda") * 0.25
    vc = torch.randn((64, 1, 16, D), generator=gen, device="cuda")
    q = torch.randn((1, heads, D), generator=gen, device="cuda")
    q[:, :, 0] = 8.0  # (a score is q k / 8)
    kc[..., 0] = 0.0
    kc[0, ..., 0] = float(np.log(rest / first))
    vc[0] += 1.0
    table = torch.cat([torch.zeros(first, dtype=torch.int32), 1 + torch.arange(rest, dtype=torch.int32) % 63]).cuda()[None].contiguous()
    i32 = lambda x: torch.tensor([x], dtype=torch.int32, device="cuda")  # noqa: E731
    out = torch.empty_like(q)
    a = wb.make_attn_args(draft_lens=i32(0), context_lens=i32(16 * (first + rest) - 1), block_tables=table, q=q, k_cache=kc,
                          v_cache=vc, out=out)
    ws = wb.alloc_workspace(wb.wisp_verify_workspace_size(a, None))
    wb.wisp_verify_attention(a, ws)
    torch.cuda.synchronize()
    assert wb.wisp_verify_get_device_status(ws) == (0, -1)
    count = torch.bincount(table[0].long(), minlength=64).double().repeat_interleave(16)  # of every key of the pool
    s = q[0].double() @ kc.view(-1, D).double().T / 8.0
    w = torch.exp(s - s.max()) * count
    ref = (w / w.sum(dim=1, keepdim=True)) @ vc.view(-1, D).double()
    assert float((out[0].double() - ref).abs().max()) <= 1e-4

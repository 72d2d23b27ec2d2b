"""The tensor-core attention where its softmax references and its chunk merge can go wrong, against the
fp64 oracle (GPU only).

The reference of a row is the maximum over its item's first 128 keys; an item with a score more than 2^64 times
past it is computed again with its true maxima.  bf16 outputs: 2e-2 absolute, as
everywhere for bf16 KV (P and the output are rounded to 8 bits; |V| is about 1 to 4 here).
"""
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
    assert err <= 2e-2, err


def _scale_keys(b, r, t0, t1, s):
    """Keys t0 .. t1 of request r times s (bf16 bits)."""
    for t in range(t0, t1):
        page = b.block_tables[r, t // 16]
        x = wl.bf16_bits_to_f32(b.k_cache[page, :, t % 16]) * np.float32(s)
        b.k_cache[page, :, t % 16] = wl.f32_to_bf16_bits(x)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("split", [False, True])  # one item per head, or chunks whose partials are merged
def test_scores_far_above_the_first_tile(D, split):
    """Keys past the first tile scaled so that scores exceed the first tile's maximum by well over 2^64
    for most rows (score sd 40 x log2 e), in the last rows' causal range too."""
    ctx, B = (3000, 2) if split else (700, 40)
    b = wl.make_batch_from_lengths("peaks", draft_lens=[5] * B, context_lens=[ctx + 7 * i for i in range(B)], Hq=32, Hkv=8,
                                   D=D, V=64, dtype="bf16", sigma=0.5, key=(170 + D, int(split)), shuffle_blocks=True)
    for r in range(0, B, 2):  # every other request: its neighbours stay ordinary
        n = int(b.context_lens[r]) + 6
        _scale_keys(b, r, 300, 340, 40.0)
        _scale_keys(b, r, n - 3, n, 40.0)
    _check(b)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("k, Hq, Hkv", [(0, 4, 4), (0, 32, 8), (4, 8, 2), (7, 32, 8), (8, 32, 8), (12, 28, 4), (15, 32, 8), (16, 32, 8)])
def test_rows_and_chunks(D, k, Hq, Hkv):
    """1 to 91 query rows per KV head (both softmax halves, one and two row groups, odd row counts in the
    merge), chunk ends on and next to tile and causal edges."""
    ctx = [0, 1, 127 - k, 128, 255, 256 + 128 - k, 2047, 2300]
    b = wl.make_batch_from_lengths("rows", draft_lens=[k] * len(ctx), context_lens=ctx, Hq=Hq, Hkv=Hkv, D=D, V=64,
                                   dtype="bf16", sigma=0.5, key=(180 + k, D), shuffle_blocks=True)
    _check(b)


def test_many_chunks():
    """One request and one KV head: over 32 chunks to merge."""
    b = wl.make_batch_from_lengths("chunks", draft_lens=[6], context_lens=[20001], Hq=4, Hkv=1, D=128, V=64, dtype="bf16",
                                   sigma=0.5, key=(190, 0))
    _check(b)


def _set_level(b, r, keys, level):
    """Component 0 of request r's `keys` such that their scores rise by about `level` in log2 (q's is 8)."""
    x = wl.f32_to_bf16_bits(np.float32([level * np.sqrt(b.D) / (8.0 * np.log2(np.e))]))[0]
    for t in keys:
        b.k_cache[b.block_tables[r, t // 16], :, t % 16, 0] = x


def _growth(b, r, t0, t1):
    """How far, in log2, each row's largest score of keys t0 .. t1 lies above that of the first 128 of them."""
    q0, n = int(b.q_row_start()[r]), int(b.draft_lens[r]) + 1
    q = wl.bf16_bits_to_f32(b.q[q0:q0 + n]).astype(np.float64).reshape(n, b.Hkv, b.Hq // b.Hkv, b.D)
    t = np.arange(t0, t1)
    k = wl.bf16_bits_to_f32(b.k_cache[b.block_tables[r, t // 16], :, t % 16]).astype(np.float64)
    s = np.einsum("nhgd,thd->nhgt", q, k) * (np.log2(np.e) / np.sqrt(b.D))
    return s.max(axis=3) - s[..., :128].max(axis=3)


@pytest.mark.parametrize("D", [64, 128])
def test_scores_above_the_first_tile_by_less(D):
    """Whole sequences whose rows all end between 2^10 and 2^60 above their reference: weights, row sums and O far
    above 1, nothing computed again."""
    B = 40
    b = wl.make_batch_from_lengths("band", draft_lens=[5] * B, context_lens=[700 + i for i in range(B)], Hq=32, Hkv=8, D=D, V=64,
                                   dtype="bf16", sigma=0.5, key=(200, D), shuffle_blocks=True)
    b.q[:, :, 0] = wl.f32_to_bf16_bits(np.float32([8.0]))[0]
    for r in range(B):
        n = int(b.context_lens[r]) + 6
        _set_level(b, r, range(5, 128, 20), (45, 30)[r % 2])
        _set_level(b, r, range(300, n - 6, 50), 65)
        g = _growth(b, r, 0, n - 6)
        assert g.min() > 10 and g.max() < 60
    _check(b)


@pytest.mark.parametrize("D", [64, 128])
def test_chunks_on_both_sides_of_the_limit(D):
    """Chunks of 256 keys (the shortest: two requests) that all reach the same level, from 0, 20, 35 and 80 below it in
    their first 128 keys: each holds a like share of the result, a quarter of them computed again."""
    b = wl.make_batch_from_lengths("sides", draft_lens=[5, 5], context_lens=[4000, 3003], Hq=32, Hkv=8, D=D, V=64,
                                   dtype="bf16", sigma=0.5, key=(201, D), shuffle_blocks=True)
    b.q[:, :, 0] = wl.f32_to_bf16_bits(np.float32([8.0]))[0]
    for r in range(2):
        n = int(b.context_lens[r])
        for i, t0 in enumerate(range(0, n - 256, 256)):
            if i % 4 != 3:
                _set_level(b, r, range(t0 + 3, t0 + 128, 20), 80 - (0, 20, 35)[i % 4])
            _set_level(b, r, range(t0 + 130, t0 + 256, 20), 80)
            g = _growth(b, r, t0, t0 + 256)
            assert (g.min() > 64) if i % 4 == 3 else (g.max() < 60)
    _check(b)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("B, ctx", [(40, 700), (1, 9000)])
def test_keys_of_minus_infinity(D, B, ctx):
    """Keys whose scores are -inf have weight zero, also where an item's first 128 keys or all of them are such."""
    b = wl.make_batch_from_lengths("inf", draft_lens=[5] * B, context_lens=[ctx + i for i in range(B)], Hq=8, Hkv=4, D=D, V=64,
                                   dtype="bf16", sigma=0.5, key=(241, D, B), shuffle_blocks=True)
    b.q[:, :, 0] = wl.f32_to_bf16_bits(np.abs(wl.bf16_bits_to_f32(b.q[:, :, 0])) + np.float32(0.1))
    for r in range(B):
        n = int(b.context_lens[r]) + 6
        for t in [*range(min(640, n // 2)), n // 2 + 1, n - 20]:
            b.k_cache[b.block_tables[r, t // 16], :, t % 16, 0] = 0xFF80
    _check(b)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("B, ctx", [(24, 8192), (2, 60000)])
def test_growing_scores_cost_a_few_passes(D, B, ctx):
    """Every item's scores pass the limit: 64 query rows, 64 tiles an item (25 where sequences are cut).  Three
    passes over the keys instead of one, and two over the values: four times an ordinary batch's time at
    most; twice that is allowed here."""
    k, Hq, Hkv = 15, 32, 8
    n, T = ctx + k + 1, B * (k + 1)
    pages = -(-n // 16)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(B)
    kc = torch.randn((B * pages, Hkv, 16, D), generator=gen, device="cuda", dtype=torch.bfloat16)
    vc = torch.randn((B * pages, Hkv, 16, D), generator=gen, device="cuda", dtype=torch.bfloat16)
    q = torch.randn((T, Hq, D), generator=gen, device="cuda", dtype=torch.bfloat16)
    table = torch.arange(B * pages, dtype=torch.int32, device="cuda").view(B, pages)
    full = lambda v: torch.full((B,), v, dtype=torch.int32, device="cuda")  # noqa: E731
    out = torch.empty_like(q)

    def timed():
        a = wb.make_attn_args(draft_lens=full(k), context_lens=full(ctx), block_tables=table, q=q, k_cache=kc, v_cache=vc, out=out)
        ws = wb.alloc_workspace(wb.wisp_verify_workspace_size(a, None))
        ms = []
        for _ in range(4):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            wb.wisp_verify_attention(a, ws)
            t1.record()
            torch.cuda.synchronize()
            ms.append(t0.elapsed_time(t1))
        assert wb.wisp_verify_get_device_status(ws) == (0, -1)
        return min(ms)

    plain = timed()
    grown = kc.view(B, pages, Hkv, 16, D)
    grown[:, torch.arange(20, pages, 50, device="cuda")] *= 40.0  # 16 keys in every 800, none in the first 128 of an item (chunks of 3200 keys)
    slow = timed()
    for r in {0, B - 1}:
        kk = kc.view(B, pages, Hkv, 16, D)[r].transpose(0, 1).reshape(Hkv, -1, D)[:, :n].double()
        vv = vc.view(B, pages, Hkv, 16, D)[r].transpose(0, 1).reshape(Hkv, -1, D)[:, :n].double()
        x = q[r * (k + 1):(r + 1) * (k + 1)].double().view(k + 1, Hkv, Hq // Hkv, D).transpose(0, 1).reshape(Hkv, -1, D)
        s = (x @ kk.transpose(1, 2) / D ** 0.5).view(Hkv, k + 1, Hq // Hkv, n)
        seen = torch.arange(n, device="cuda")[None] <= ctx + torch.arange(k + 1, device="cuda")[:, None]
        s = s.masked_fill(~seen[None, :, None, :], float("-inf")).softmax(dim=-1)
        ref = (s.view(Hkv, -1, n) @ vv).view(Hkv, k + 1, Hq // Hkv, D).transpose(0, 1).reshape(k + 1, Hq, D)
        assert float((out[r * (k + 1):(r + 1) * (k + 1)].double() - ref).abs().max()) <= 3e-2
    print(f"D {D}, B {B}, context {ctx}: {plain:.3f} ms, with scores past the limit {slow:.3f} ms")
    assert slow < 8 * plain, (plain, slow)

"""Page reservation where the cluster's work split can go wrong, against the plain-Python model, bit for
bit: more requests than one scan round (1024) and than the cluster's warps (256), rows longer than one
load round (128 pages), missing pages anywhere in a row, refused requests among served ones, and a row count that
the lengths do not add up to."""
import numpy as np
import pytest
import torch

from oracle import kv as model

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B, ctx_hi, k_hi, hole, bad, short", [
    (1, 5000, 3, 0.0, 0.0, 0), (3, 4100, 40, 0.3, 0.0, 0), (257, 300, 5, 0.1, 0.05, 0), (1024, 64, 3, 0.2, 0.02, 0),
    (1500, 90, 4, 0.2, 0.02, 0), (2600, 40, 2, 0.5, 0.01, 700)])
def test_reserve(B, ctx_hi, k_hi, hole, bad, short):
    from paper_2601_11652_gb300 import binding as wb, build
    build.build()
    rng = np.random.default_rng(B + k_hi)
    ctx = rng.integers(0, ctx_hi, size=B).tolist()
    draft = rng.integers(0, k_hi + 1, size=B).tolist()
    pages = [(c + k + 1 + 15) // 16 for c, k in zip(ctx, draft)]
    mb, nb = max(pages) + 2, sum(pages) + 5
    perm = rng.permutation(nb).tolist()
    tables = [[-1] * mb for _ in range(B)]
    for r in range(B):
        for b in range((ctx[r] + 15) // 16):
            if rng.random() >= hole:
                tables[r][b] = perm.pop()
    for r in range(B):
        if rng.random() < bad:
            tables[r][0] = nb + 3  # a page id outside the pool
    F = max(0, len(perm) - short)
    stack = perm + [-1] * (nb - len(perm))
    T, Hkv, D = sum(draft) + B, 1, 64
    kn, vn = (rng.standard_normal((T, Hkv, D)).astype(np.float32) for _ in range(2))
    kc, vc = (np.zeros((nb, Hkv, 16, D), np.float32) for _ in range(2))
    dev = lambda a, dt=None: torch.tensor(np.asarray(a), dtype=dt, device="cuda")  # noqa: E731
    g = dict(draft_lens=dev(draft, torch.int32), context_lens=dev(ctx, torch.int32), block_tables=dev(tables, torch.int32),
             free_blocks=dev(stack, torch.int32), free_count=dev([F], torch.int32), k_cache=dev(kc), v_cache=dev(vc),
             k_new=dev(kn), v_new=dev(vn))
    args = wb.make_kv_args(**g)
    ws = wb.alloc_workspace(wb.wisp_kv_workspace_size(args))
    wb.wisp_kv_reserve_append(args, ws)
    torch.cuda.synchronize()
    code, _ = wb.wisp_verify_get_device_status(ws)
    F1, codes = model.reserve_append(tables, stack, F, ctx, draft, nb, kn, vn, kc, vc)
    errs = {c for c in codes if c}
    assert code in errs if errs else code == 0
    assert np.array_equal(g["block_tables"].cpu().numpy(), np.asarray(tables, np.int32))
    assert int(g["free_count"].item()) == F1
    assert np.array_equal(g["k_cache"].cpu().numpy(), kc) and np.array_equal(g["v_cache"].cpu().numpy(), vc)


@pytest.mark.parametrize("B, extra", [(1, 1), (70, 5000), (1500, 300), (40, -3)])
def test_row_count_that_disagrees(B, extra):
    """total_q_rows past the sum of the lengths, or short of it: flagged; the rows that belong to a request are written
    and no other, whatever the workspace held."""
    from paper_2601_11652_gb300 import binding as wb, build
    build.build()
    rng = np.random.default_rng(B)
    ctx = rng.integers(0, 60, size=B).tolist()
    draft = rng.integers(0, 4, size=B).tolist()
    pages = [(c + k + 1 + 15) // 16 for c, k in zip(ctx, draft)]
    mb, nb = max(pages), sum(pages) + 5
    perm = rng.permutation(nb).tolist()
    tables = [[perm.pop() if b < (ctx[r] + 15) // 16 else -1 for b in range(mb)] for r in range(B)]
    F = len(perm)
    stack = perm + [-1] * (nb - len(perm))
    T, Hkv, D = sum(draft) + B, 2, 64
    kn, vn = (rng.standard_normal((max(T, T + extra), Hkv, D)).astype(np.float32) for _ in range(2))
    kc, vc = (np.zeros((nb, Hkv, 16, D), np.float32) for _ in range(2))
    dev = lambda a, dt=None: torch.tensor(np.asarray(a), dtype=dt, device="cuda")  # noqa: E731
    g = dict(draft_lens=dev(draft, torch.int32), context_lens=dev(ctx, torch.int32), block_tables=dev(tables, torch.int32),
             free_blocks=dev(stack, torch.int32), free_count=dev([F], torch.int32), k_cache=dev(kc), v_cache=dev(vc),
             k_new=dev(kn), v_new=dev(vn))
    args = wb.make_kv_args(**g, total_q_rows=T + extra)
    ws = wb.alloc_workspace(wb.wisp_kv_workspace_size(args))
    ws.zero_()  # left-over words that name request 0, position 0
    wb.wisp_kv_reserve_append(args, ws)
    torch.cuda.synchronize()
    assert wb.wisp_verify_get_device_status(ws)[0] == 1
    model.reserve_append(tables, stack, F, ctx, draft, nb, kn[:T], vn[:T], kc, vc)
    if extra < 0:  # the last rows are past the caller's count
        for x in range(T + extra, T):
            r = int(np.searchsorted(np.cumsum(np.asarray(draft) + 1), x, side="right"))
            pos = ctx[r] + x - (sum(draft[:r]) + r)
            kc[tables[r][pos // 16], :, pos % 16] = vc[tables[r][pos // 16], :, pos % 16] = 0.0
    assert np.array_equal(g["k_cache"].cpu().numpy(), kc) and np.array_equal(g["v_cache"].cpu().numpy(), vc)

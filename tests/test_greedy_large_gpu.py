"""The greedy variant in level-major order (batches above 128 MiB of logits) against the oracle: walks that end
at every level, ties, rows without a finite logit, draft tokens outside the vocabulary, fp32 and an
unaligned vocabulary (GPU only; integers, exact)."""
import numpy as np
import pytest
import torch

from tests.test_greedy import _Batch, wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype, B, k_hi, V", [("bf16", 300, 3, 128256), ("bf16", 1100, 8, 16001), ("f32", 90, 6, 128256),
                                               ("f32", 2300, 2, 9999)])
def test_level_major(oracle_mod, dtype, B, k_hi, V):
    from paper_2601_11652_gb300 import binding as wb, build
    build.build()
    rng = np.random.default_rng(B)
    k = rng.integers(0, k_hi + 1, size=B).astype(np.int32)
    T = int(k.sum()) + B
    assert T * V * (2 if dtype == "bf16" else 4) > 128 << 20
    z = np.round(rng.standard_normal((T, V), dtype=np.float32) * 4) / 4  # coarse values: ties at the maximum
    qs = np.concatenate([[0], np.cumsum(k + 1)])
    z[qs[5]] = -np.inf   # row 0 of request 5 has no finite logit
    toks = []
    for r in range(B):
        for i in range(int(k[r])):
            toks.append(int(np.argmax(z[qs[r] + i])) if rng.random() < 0.7 else int(rng.integers(V)))
    ds = np.concatenate([[0], np.cumsum(k)])
    r_bad = int(np.nonzero(k > 0)[0][3])
    toks[ds[r_bad]] = V + 7
    b = _Batch(wl.f32_to_bf16_bits(z) if dtype == "bf16" else z, k, toks, dtype)
    ref = oracle_mod.accept_greedy(b)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    lg = dev(b.logits.view(np.int16)).view(torch.bfloat16) if dtype == "bf16" else dev(b.logits)
    none = torch.empty(0, dtype=torch.float32, device="cuda")
    out = {n: torch.full((B,), -7, dtype=torch.int32, device="cuda") for n in ("accepted_len", "next_token")}
    args = wb.make_accept_args(draft_lens=dev(b.draft_lens), target_logits=lg, draft_tokens=dev(b.draft_tokens),
                               draft_probs=none, accept_uniforms=none, sample_uniforms=none, **out)
    ws = wb.alloc_workspace(wb.wisp_verify_workspace_size(None, args))
    for _ in range(3):  # the same workspace again: the planner clears the launch's state
        wb.wisp_verify_accept_greedy(args, ws)
    torch.cuda.synchronize()
    assert wb.wisp_verify_get_device_status(ws)[0] in (3, 4)
    good = np.ones(B, bool)
    good[[5, r_bad]] = False
    assert np.array_equal(out["accepted_len"].cpu().numpy()[good], ref["accepted_len"][good])
    assert np.array_equal(out["next_token"].cpu().numpy()[good], ref["next_token"][good])
    assert np.all(out["next_token"].cpu().numpy()[~good] == -1)

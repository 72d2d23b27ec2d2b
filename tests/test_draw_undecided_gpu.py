"""GPU: draw slices with many elements whose q is p to a rounding, so that the fp32 test leaves the sign of p - q
open: up to the number a slice keeps (64; 8 in the fixed scratch), one more, and all of a row (the residual's whole mass
is then rounding of q).  The fp64 oracle's tokens exactly, outside the windows that every comparison logs."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_11652_gb300 import workload as wl
from tests.gpu_util import compare_accept

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2601_11652_gb300 import build
    build.build()


@pytest.mark.parametrize("noalloc", [False, True])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("n", [1, 8, 9, 64, 65, 500, 1999])
def test_undecided_elements(n, dtype, noalloc):
    from paper_2601_11652_gb300 import binding as wb
    from paper_2601_11652_gb300.device_batch import DeviceBatch
    B, V = 12, 2000  # one draw slice
    rng = np.random.default_rng([n, V])
    b = wl.make_batch_from_lengths("undecided", draft_lens=[1] * B, context_lens=[3] * B, Hq=8, Hkv=2, D=128, V=V,
                                   dtype=dtype, sigma=0.5, key=(77, n))
    qs, ds = b.q_row_start(), b.draft_start()
    for r in range(B):
        p = oracle.row_softmax(b.logits[qs[r]], b.dtype)
        y = int(b.draft_tokens[ds[r]])
        q = p * rng.choice([0.5, 1.5], V)
        equal = rng.permutation(np.delete(np.arange(V), y))[:n]
        q[equal] = p[equal]
        q[y] = 2.0 * p[y] + 0.1  # rejected: u is above p / q
        b.draft_probs[ds[r]] = q.astype(np.float32)
        b.accept_uniforms[ds[r]] = np.float32(0.99)
    ref = oracle.accept(b)
    assert np.all(ref["accepted_len"] == 0)
    db = DeviceBatch.from_host(b)
    wb.wisp_verify_accept_noalloc(db.accept_args) if noalloc else db.accept()
    torch.cuda.synchronize()
    got = db.results()
    if not noalloc:
        assert db.device_status() == (0, -1)
    compared, _ = compare_accept(b, got["accepted_len"], got["next_token"], ref)
    assert compared >= B - 2

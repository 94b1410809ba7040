"""The one-call entry points queue mask and attention without reading the mask's pair count back where
the key lists are small: their outputs are those of the same calls on a mask built beforehand."""
import pytest
import torch

from helpers import make_inputs
from paper_2607_21927_gb300 import ris

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 40, 3001, 8300])
@pytest.mark.parametrize("mode,d,S,W,A,sampler", [
    (0, 0.01, 3, 1, 0, 0), (1, 0.1, 2, 1, 4, 0), (0, 0.02, 2, 300, 0, 1), (0, 0.3, 2, 1, 0, 0)],
    ids=["gather", "blocks", "window_draws", "tiles"])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_one_call_equals_prebuilt_mask(N, mode, d, S, W, A, sampler, dtype):
    q, k, v = make_inputs(N, 6, 2, 128, dtype=dtype, seed=N + S, outliers=True)[0]
    seeds, opts, rope = list(range(S)), ris.mask_opts(W, A, sampler=sampler), ris.rope_cfg(3, 1e6, 1024)
    for per_seed, fn in ((False, ris.ris_sparse_attention_fwd), (True, ris.ris_ensemble_batch)):
        if per_seed and dtype == torch.float32 and N > 4000:
            continue  # the sized path once is enough
        out, lse = fn(q, k, v, mode, d, seeds, rope=rope, opts=opts, out_dtype=torch.float32, return_lse=True)
        with ris.ris_mask_generate(N, 2, mode, d, seeds, opts, per_seed=per_seed) as m:
            ref, ref_lse = ris.ris_attention_masked(m, q, k, v, rope, out_dtype=torch.float32, return_lse=True)
        assert torch.equal(out, ref) and torch.equal(lse, ref_lse)


@pytest.mark.parametrize("mode,d,A", [(0, 0.01, 0), (1, 0.01, 4)], ids=["stochastic", "blocks"])
def test_seeds_given_twice_count_once(mode, d, A):
    """Twenty times the same seed keep what one keeps, and the one call takes the design of that mask."""
    q, k, v = make_inputs(3001, 8, 2, 64, seed=9)[0]
    seeds, opts, rope = [7] * 20, ris.mask_opts(1, A), ris.rope_cfg(3, 1e6, 1024)
    out = ris.ris_sparse_attention_fwd(q, k, v, mode, d, seeds, rope=rope, opts=opts, out_dtype=torch.float32)
    with ris.ris_mask_generate(3001, 2, mode, d, seeds, opts) as m:
        assert ris.ris_attention_design(m, torch.bfloat16, 64) == 0
        assert torch.equal(out, ris.ris_attention_masked(m, q, k, v, rope, out_dtype=torch.float32))

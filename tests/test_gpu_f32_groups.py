"""The fp32 gather at every group size its kernels are built for, at rows around its 16-key steps, both
head dims, list and dense masks, fp32 and bf16 outputs."""
import numpy as np
import pytest
import torch

from helpers import check_f32_path, make_inputs, to_np
from test_gpu_attention import run_gpu, run_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hq,Hkv", [(1, 1), (4, 2), (3, 1), (8, 2), (5, 1), (12, 2), (7, 1), (8, 1)])
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("N,mode,d", [(1, 2, 1.0), (35, 2, 1.0), (150, 0, 0.2)])
def test_f32_groups(Hq, Hkv, D, N, mode, d):
    (q, k, v), (qn, kn, vn) = make_inputs(N, Hq, Hkv, D, dtype=torch.float32, seed=N + Hq)
    out, lse = run_gpu(q, k, v, mode, d, [1, 2], 3, 1e4, 64)
    ref, ref_lse = run_oracle(qn, kn, vn, mode, d, [1, 2], 3, 1e4, 64)
    check_f32_path(to_np(out), ref)
    np.testing.assert_allclose(to_np(lse).T, ref_lse, rtol=1e-5, atol=1e-5)
    # the same sums rounded to bf16: half an ulp, and one flip of the rounding by the fp32 error
    half, _ = run_gpu(q, k, v, mode, d, [1, 2], 3, 1e4, 64, out_dtype=torch.bfloat16)
    assert (np.abs(to_np(half) - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-5).all()


@pytest.mark.parametrize("Hq,Hkv,D", [(2, 2, 64), (4, 2, 128), (12, 2, 128)])
def test_f32_infinite_values_stay_infinite(Hq, Hkv, D):
    """A row whose own value is infinite comes out infinite, whatever the row's length leaves of the kernel's
    last step; rows and channels without one come out as they are."""
    N = 70
    (q, k, v), _ = make_inputs(N, Hq, Hkv, D, dtype=torch.float32, seed=D)
    ref, _ = run_gpu(q, k, v, 2, 1.0, [1], 0, 1e4, 64)
    keys = [13, 34, 36, 69]
    for c, j in enumerate(keys):
        v[j, :, c] = float("inf") if c % 2 == 0 else -float("inf")
    out, lse = run_gpu(q, k, v, 2, 1.0, [1], 0, 1e4, 64)
    for c, j in enumerate(keys):
        assert torch.equal(out[:j, :, c], ref[:j, :, c])
        assert (out[j:, :, c] == v[j, 0, c]).all()
    assert torch.equal(out[:, :, len(keys):], ref[:, :, len(keys):]) and torch.isfinite(lse).all()

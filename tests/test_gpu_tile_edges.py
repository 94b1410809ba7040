"""The tile kernel at the edges of its tiles: one to five key tiles (either group of softmax warps
without tiles, with one or several), full and single-row last tiles, both head dims, odd and even
query groups, dense and masked, rotated and as-given inputs."""
import numpy as np
import pytest
import torch

from helpers import check_bf16_path, make_inputs, to_np
from test_gpu_attention import run_gpu, run_oracle
from paper_2607_21927_gb300 import ris

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 2, 127, 128, 129, 256, 257, 385, 513, 640])
@pytest.mark.parametrize("Hq,Hkv,D", [(6, 2, 128), (3, 1, 128), (4, 2, 64)])
@pytest.mark.parametrize("mode,d,kind", [(2, 1.0, 3), (0, 0.4, 3), (2, 1.0, 0)], ids=["dense", "masked", "dense_unrotated"])
def test_tile_edges(N, Hq, Hkv, D, mode, d, kind):
    (q, k, v), (qn, kn, vn) = make_inputs(N, Hq, Hkv, D, seed=N + D, outliers=True)
    with ris.ris_mask_generate(N, Hkv, mode, d, [3]) as m:
        assert ris.ris_attention_design(m, torch.bfloat16, D) == 2
    out, lse = run_gpu(q, k, v, mode, d, [3], kind, 1e4, 256)
    ref, ref_lse = run_oracle(qn, kn, vn, mode, d, [3], kind, 1e4, 256)
    check_bf16_path(to_np(out), ref)
    np.testing.assert_allclose(to_np(lse).T, ref_lse, rtol=0, atol=2e-2)


@pytest.mark.parametrize("mode,d", [(2, 1.0), (0, 0.4)], ids=["dense", "masked"])
@pytest.mark.parametrize("Hq,Hkv,D", [(6, 2, 128), (4, 2, 64)])
def test_row_maximum_grows_in_every_tile(mode, d, Hq, Hkv, D):
    """Scores that rise by about 10 (log2) from each key tile to the next: O is rescaled in every tile
    by both groups, every other row only (the queries of even rows point the other way, so theirs fall)."""
    N = 900
    (q, k, v), _ = make_inputs(N, Hq, Hkv, D, seed=D)
    u = torch.ones(D, device=q.device) / D**0.5
    sign = 1.0 - 2.0 * (torch.arange(N, device=q.device) % 2 == 0).float()
    q = (0.3 * q.float() + 8.0 * sign[:, None, None] * u).to(torch.bfloat16)
    step = 7.0 * D**0.5 / 8.0  # of the keys' component along u: a score step of 7 (natural log)
    k = (0.3 * k.float() + step * (torch.arange(N, device=q.device) // 128).float()[:, None, None] * u).to(torch.bfloat16)
    qn, kn, vn = (to_np(x).astype(np.float64) for x in (q, k, v))
    out, lse = run_gpu(q, k, v, mode, d, [3], 0, 1e4, 256)
    ref, ref_lse = run_oracle(qn, kn, vn, mode, d, [3], 0, 1e4, 256)
    check_bf16_path(to_np(out), ref)
    np.testing.assert_allclose(to_np(lse).T, ref_lse, rtol=0, atol=2e-2)

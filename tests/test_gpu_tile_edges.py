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

"""The tile kernel at the edges of its tiles: one to five key tiles (either group of softmax warps
without tiles, with one or several), full and single-row last tiles, both head dims, dense and masked,
rotated and as-given inputs. At head dim 128 the two CTAs of a cluster take two heads of an even query group
(4 / 2) or two query tiles of a head of an odd one (6 / 2, 3 / 1); at head dim 64 there are no clusters."""
import numpy as np
import pytest
import torch

from helpers import check_bf16_path, make_inputs, to_np
from test_gpu_attention import run_gpu, run_oracle
from paper_2607_21927_gb300 import ris

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 2, 127, 128, 129, 256, 257, 385, 513, 640])
@pytest.mark.parametrize("Hq,Hkv,D", [(4, 2, 128), (6, 2, 128), (3, 1, 128), (4, 2, 64)])
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
@pytest.mark.parametrize("Hq,Hkv,D", [(4, 2, 128), (6, 2, 128), (4, 2, 64)])
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


@pytest.mark.parametrize("mode,d,W,design", [(0, 0.5, 1, 2), (2, 1.0, 1, 2), (0, 0.01, 300, 4)], ids=["masked", "dense", "split"])
def test_even_groups_on_row_ranges(mode, d, W, design):
    """Row ranges that start and end inside 128-row tiles, on the whole layer's tensors and on local rows,
    with two heads of a group per cluster: bit for bit the rows of the whole layer. The power-of-two scales of
    the score operands follow from the largest pair norm of the queries given, so every row gets
    the same largest pair."""
    N, Hq, Hkv, D = 1700, 12, 2, 128
    q, k, v = make_inputs(N, Hq, Hkv, D, seed=31)[0]
    q[:, 0, 0], q[:, 0, D // 2] = 12.0, 0.0
    rope = ris.rope_cfg(3, 1e6, 256)
    with ris.ris_mask_generate(N, Hkv, mode, d, [4], ris.mask_opts(W)) as m:
        assert ris.ris_attention_design(m, torch.bfloat16, D) == design
        whole, lse = ris.ris_attention_masked(m, q, k, v, rope=rope, out_dtype=torch.float32, return_lse=True)
        parts = torch.full_like(whole, float("nan"))
        edges = [0, 1, 127, 300, 301, 512, 1153, N]
        for r0, r1 in zip(edges[:-1], edges[1:]):
            ris.ris_attention_masked_rows(m, r0, r1, q, k, v, parts, rope=rope)
            o, part_lse = ris.ris_attention_masked_local(m, r0, r1, q[r0:r1].clone(), k, v, rope=rope,
                                                         out_dtype=torch.float32, return_lse=True)
            assert torch.equal(o, whole[r0:r1]) and torch.equal(part_lse, lse[:, r0:r1])
        torch.cuda.synchronize()
        ris.ris_device_status()
        assert torch.equal(parts, whole)

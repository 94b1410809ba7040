"""A call on a few local rows of a long sequence reads all keys and values with the whole chip."""
import pytest
import torch

from helpers import make_inputs
from paper_2607_21927_gb300 import ris

pytestmark = pytest.mark.gpu


def _us(fn, n=20):
    fn()
    best = float("inf")
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(n):
            fn()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) / n * 1e3)
    return best


@pytest.mark.parametrize("Hq,Hkv", [(12, 2), (8, 8)])
def test_fewer_local_rows_take_no_longer(Hq, Hkv):
    """The passes over k and v are the same whatever the rows, the rest grows with them: 8 rows of 65,536 take
    no longer than 1,024. (With the grid of the first pass sized by the rows they took 6 to 14 times as long.)"""
    N, rope = 65536, ris.rope_cfg(3, 1e6, 32768)
    q, k, v = make_inputs(N, Hq, Hkv, 128, seed=3)[0]
    with ris.ris_mask_generate(N, Hkv, 0, 0.01, [5]) as m:
        assert ris.ris_attention_design(m, torch.bfloat16, 128) == 0
        t = {}
        for rows in (8, 1024):
            part = q[N - rows:].clone()
            t[rows] = _us(lambda: ris.ris_attention_masked_local(m, N - rows, N, part, k, v, rope=rope))
    print(f"{Hq}/{Hkv}: 8 rows {t[8]:.1f} us, 1,024 rows {t[1024]:.1f} us")
    assert t[8] <= 1.1 * t[1024]

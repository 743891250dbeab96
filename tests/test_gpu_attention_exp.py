"""The attention kernel's exponentials: scores over the whole
range of the exponent, keys that must not count, and NaN, at every position of a group of sixteen keys."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2607_19438_b200 import binding as qg, synth
from tests import util

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
def test_scores_over_the_whole_range(d):
    """Scores spread over +-200 in the exponent: most keys underflow, the rest span every binade."""
    S, Hq, Hkv = 300, 2, 1
    rng = np.random.default_rng(d)
    Q, K, V = (synth.f32_to_bf16_bits((rng.standard_normal((S, h * d)) * a).astype(np.float32)) for h, a in ((Hq, 6.0), (Hkv, 6.0), (Hkv, 1.0)))
    out = qg.prefill_attention(util.dev_bf16(Q), util.dev_bf16(K), util.dev_bf16(V), Hq, Hkv, d, causal=True)
    qg.poll_status()
    ref = orc.attention(Q, K, V, Hq, Hkv, d, causal=True)
    util.assert_close(util.host_bf16_f64(out), ref, "wide scores")


@pytest.mark.parametrize("d", [64, 128])
def test_a_nan_key_reaches_the_rows_that_see_it_and_no_others(d):
    S, H = 160, 1
    rng = np.random.default_rng(d + 1)
    Q, K, V = (torch.from_numpy(rng.standard_normal((S, H * d)).astype(np.float32)).cuda().to(torch.bfloat16) for _ in range(3))
    for key in list(range(32, 48)) + [128, 129, 143]:
        Kn = K.clone()
        Kn[key] = float("nan")
        out = qg.prefill_attention(Q, Kn, V, H, H, d, causal=True)
        qg.poll_status()
        assert bool(torch.isnan(out[key:]).all()) and not bool(torch.isnan(out[:key]).any()), key


@pytest.mark.parametrize("d", [64, 128])
def test_scores_of_minus_infinity_count_as_nothing(d):
    """Keys at minus infinity against a positive query: weight zero wherever the other keys are finite, and zero output, not a
    mean of values, for rows that see nothing else."""
    S = 40
    Q = torch.ones((S, d), device="cuda").to(torch.bfloat16)
    K = torch.zeros((S, d), device="cuda").to(torch.bfloat16)
    V = torch.randn((S, d), device="cuda").to(torch.bfloat16)
    K[:18, 0] = float("-inf")
    out = qg.prefill_attention(Q, K, V, 1, 1, d, causal=True)
    qg.poll_status()
    assert float(out[:18].abs().max()) == 0.0
    ref = V[18:].double().cumsum(0) / torch.arange(1, S - 17, device="cuda")[:, None]
    assert float((out[18:].double() - ref).abs().max()) < 2e-2

"""Negative distortion weights and a negative head sensitivity against the oracle.

With lambda_Z or lambda_M negative a node's distortion may be negative, and
omega R D then bounds no split's utility from above; the same goes for a
negative omega.  The trees must still be built as far as the budget reaches:
most keys are 0 here (clamped), so the selection runs into the tied ops at 0
and takes splits far below the roots.  The weights have one sign, so that D
has no cancellation and compares at the usual tolerance.
"""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2608_07001_gb300 import synth
from tests import parity as P

pytestmark = pytest.mark.gpu

LONG = [129, 3, 160, 161, 255, 40, 289, 513]   # slots above and below the unit kernel's 128 tokens


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()
    assert torch.cuda.is_available()


@pytest.mark.parametrize("lz,lm,om", [(-0.25, -0.75, 1.0), (-0.25, 0.0, 1.0), (0.0, -0.75, 1.0), (0.25, 0.75, -1.0)])
@pytest.mark.parametrize("dtype,d,lens", [("bf16", 64, None), ("fp32", 128, None), ("bf16", 128, LONG), ("fp32", 64, LONG)])
def test_negative_weights_match_the_oracle(dtype, d, lens, lz, lm, om):
    G = 1 if lens else 2
    w = dataclasses.replace(synth.WORKLOADS["small"], L=1, G=G, Hq=4 * G, d=d)
    x = synth.make_inputs(w, T=sum(lens) + 32 if lens else 700, W=8)
    K, V, Q = x.K, x.V, x.Q
    if dtype == "fp32":
        K, V, Q = K.float(), V.float(), Q.float()
    kw = dict(lambda_Z=lz, lambda_M=lm, omega=np.full((1, G), om, dtype=np.float32))
    if lens:
        kw["slot_starts"] = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    B = G * K.shape[2] // 4
    g = P.run_gpu(K, V, Q, B, w.rope_base, **kw)
    o = P.run_oracle(K, V, Q, B, w.rope_base, **kw)
    below = o["split_sel"].astype(bool) & (o["trees"].nodes["parent"] >= 0)
    assert below.sum() > B // 2, "the budget reaches below the roots"
    P.compare(g, o, torch.float32 if dtype == "fp32" else torch.bfloat16)

"""Slot lengths at the unit kernel's class edges against the oracle.

The unit kernel has an instance for slots of up to 36, 64 and 128 tokens, and
classes too small to fill the GPU share a launch: with no short slots beside
the edge lengths every unit runs on the 128-token instance, with 200 of them
the 36-token class joins the 64-token one, with 340 every class has its own
launch.  The inputs cover the three ways the probe weights are formed (by the
score pass; on mma.sync, above 256 probe rows per KV head; in fp32).
"""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2608_07001_gb300 import synth
from tests import parity as P

pytestmark = pytest.mark.gpu

EDGES = [36, 1, 128, 37, 2, 64, 3, 65, 35, 127, 63, 17]


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()
    assert torch.cuda.is_available()


@pytest.mark.parametrize("fill", [0, 200, 340])
@pytest.mark.parametrize("dtype,d,gq,W", [("bf16", 64, 4, 8), ("bf16", 128, 8, 40), ("fp32", 128, 2, 8)])
def test_class_edges_match_the_oracle(dtype, d, gq, W, fill):
    lens = EDGES + [1 + i % 3 for i in range(fill)]
    w = dataclasses.replace(synth.WORKLOADS["small"], L=1, G=1, Hq=gq, d=d)
    x = synth.make_inputs(w, T=sum(lens) + 32, W=W)
    K, V, Q = x.K, x.V, x.Q
    if dtype == "fp32":
        K, V, Q = K.float(), V.float(), Q.float()
    slots = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    B = K.shape[2] // 3
    g = P.run_gpu(K, V, Q, B, w.rope_base, slot_starts=slots)
    o = P.run_oracle(K, V, Q, B, w.rope_base, slot_starts=slots)
    P.compare(g, o, torch.float32 if dtype == "fp32" else torch.bfloat16)


@pytest.mark.parametrize("lam", [0.0, 0.002, 1.0])
@pytest.mark.parametrize("dtype,d", [("bf16", 64), ("fp32", 128)])
def test_cut_bounds_match_the_oracle(dtype, d, lam):
    # A cut is left out when D + lambda_kappa kh is below the best cut found: with
    # lambda_kappa 0 none is, at 1 nearly all are, at 0.002 some nodes keep a few
    # and compare them with the extraction.
    w = dataclasses.replace(synth.WORKLOADS["small"], L=1, G=2, Hq=4, d=d)
    x = synth.make_inputs(w, T=700, W=16)
    K, V, Q = x.K, x.V, x.Q
    if dtype == "fp32":
        K, V, Q = K.float(), V.float(), Q.float()
    B = 2 * 700 // 4
    g = P.run_gpu(K, V, Q, B, w.rope_base, lambda_kappa=lam)
    o = P.run_oracle(K, V, Q, B, w.rope_base, lambda_kappa=lam)
    P.compare(g, o, torch.float32 if dtype == "fp32" else torch.bfloat16)


@pytest.mark.parametrize("last", [1, 2])   # 8192 ops at most (one block selects them), 8193
@pytest.mark.parametrize("ratio", [0.5, 3, 60])   # everything fits; splits; not even every Add
def test_small_selection_matches_the_oracle(last, ratio):
    lens = [64] * 126 + [last]
    w = dataclasses.replace(synth.WORKLOADS["small"], L=1, G=1, Hq=1, d=64)
    x = synth.make_inputs(w, T=sum(lens) + 32, W=8)
    slots = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    B = int(sum(lens) / ratio) + 32
    g = P.run_gpu(x.K, x.V, x.Q, B, w.rope_base, slot_starts=slots)
    o = P.run_oracle(x.K, x.V, x.Q, B, w.rope_base, slot_starts=slots)
    P.compare(g, o, torch.bfloat16)


@pytest.mark.parametrize("n", [1, 7, 8, 9, 33, 34, 35, 36])
def test_probe_weight_tiles_end_at_the_slot(n):
    # 320 probe rows per KV head: the unit kernel forms the probe weights itself, in tiles of
    # 8 tokens; with 340 slots the 36-token class runs on its own instance, whose last tile
    # has rows past the slot (and, above 32 tokens, past the instance's 36)
    lens = [n] * 40 + [1 + i % 3 for i in range(300)]
    w = dataclasses.replace(synth.WORKLOADS["small"], L=1, G=1, Hq=8, d=128)
    x = synth.make_inputs(w, T=sum(lens) + 32, W=40)
    slots = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    B = x.K.shape[2] // 3
    g = P.run_gpu(x.K, x.V, x.Q, B, w.rope_base, slot_starts=slots)
    o = P.run_oracle(x.K, x.V, x.Q, B, w.rope_base, slot_starts=slots)
    P.compare(g, o, torch.bfloat16)


@pytest.mark.parametrize("k_cand", [16, 3])
@pytest.mark.parametrize("lam", [0.0, 0.05])
@pytest.mark.parametrize("dtype,d", [("bf16", 64), ("fp32", 128)])
def test_tied_cuts_take_the_smallest(dtype, d, lam, k_cand):
    # V = 0 and lambda_Z = 0: every D is exactly 0 and the curvature of the zero trajectory
    # takes few values, so the rewards, and with them the cuts, tie; neither the cut that is
    # evaluated first nor a bound may move the choice from the smallest position
    lens = [36, 2, 3, 5, 128, 37, 64, 65, 17, 129, 300]
    w = dataclasses.replace(synth.WORKLOADS["small"], L=1, G=1, Hq=4, d=d)
    x = synth.make_inputs(w, T=sum(lens) + 32, W=8)
    K, V, Q = x.K, torch.zeros_like(x.V), x.Q
    if dtype == "fp32":
        K, V, Q = K.float(), V.float(), Q.float()
    kw = dict(lambda_Z=0.0, lambda_kappa=lam, k_cand=k_cand,
              slot_starts=np.concatenate([[0], np.cumsum(lens)]).astype(np.int32))
    B = K.shape[2] // 2
    g = P.run_gpu(K, V, Q, B, w.rope_base, **kw)
    o = P.run_oracle(K, V, Q, B, w.rope_base, **kw)
    assert not o["trees"].nodes["D"].any()
    P.compare(g, o, torch.float32 if dtype == "fp32" else torch.bfloat16)


@pytest.mark.parametrize("lam", [0.0, 1e-4, 1e-3])
@pytest.mark.parametrize("k_cand", [16, 5, 0])
@pytest.mark.parametrize("dtype,d,gq,W", [("bf16", 64, 4, 8), ("bf16", 128, 8, 40), ("fp32", 128, 2, 8)])
def test_open_cuts_match_the_oracle(dtype, d, gq, W, k_cand, lam):
    # Little or no curvature reward leaves every cut open: nodes evaluate all of them at once,
    # as many nodes at a time as fit the 19 rows (16 candidates, the midpoint, the extraction
    # and a root itself fill them), in every slot class
    lens = EDGES + [4, 5, 19, 20, 21, 40, 100] + [1 + i % 5 for i in range(40)]
    w = dataclasses.replace(synth.WORKLOADS["small"], L=1, G=1, Hq=gq, d=d)
    x = synth.make_inputs(w, T=sum(lens) + 32, W=W)
    K, V, Q = x.K, x.V, x.Q
    if dtype == "fp32":
        K, V, Q = K.float(), V.float(), Q.float()
    kw = dict(lambda_kappa=lam, k_cand=k_cand, slot_starts=np.concatenate([[0], np.cumsum(lens)]).astype(np.int32))
    B = K.shape[2] // 3
    g = P.run_gpu(K, V, Q, B, w.rope_base, **kw)
    o = P.run_oracle(K, V, Q, B, w.rope_base, **kw)
    P.compare(g, o, torch.float32 if dtype == "fp32" else torch.bfloat16)


@pytest.mark.parametrize("dtype,d", [("bf16", 64), ("fp32", 128)])
@pytest.mark.parametrize("max_len", [36, 64, 128])
def test_no_reward_scans_a_node_once_per_direction(dtype, d, max_len):
    # without a curvature reward no cut can rule another out: none is evaluated ahead of the
    # others, which would sweep the node's tokens a second time
    lens = [1 + (7 * i) % max_len for i in range(120)]
    w = dataclasses.replace(synth.WORKLOADS["small"], L=1, G=1, Hq=4, d=d)
    x = synth.make_inputs(w, T=sum(lens) + 32, W=8)
    K, V, Q = x.K, x.V, x.Q
    if dtype == "fp32":
        K, V, Q = K.float(), V.float(), Q.float()
    slots = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    g = P.run_gpu(K, V, Q, K.shape[2] // 4, w.rope_base, lambda_kappa=0.0, slot_starts=slots)
    ex = g["export"]
    n = ex["b"] - ex["a"]
    _, _, work = g["comp"].ctx.gracekv_stats()
    evaluated = (ex["nchild"] > 0) | (n == 1)   # single tokens: a root's own row
    assert work["scan_steps"] <= 2 * int(n[evaluated].sum()), work

"""The walk of a thread block cluster per sequence (small batches) and the walk of one block per sequence (large ones) give
the same bits, so a batch may be split at will: checked at the edges of the clusters' shapes (a row of exactly so many tiles,
one entry more), with rows on 16-byte boundaries, NaN and far-off rows; and against the oracle with rows off them.  (Other
rows, rules and trees in large batches: test_gpu_walk_routes.py.)"""
import numpy as np
import pytest
import torch

import oracle
import workloads
from tests.parity import Tally, compare_verify
from tests.test_gpu_parity import _np

pytestmark = pytest.mark.gpu


def _drafted(B, V, dtype, branching, seed, off=0, draft_sigma=2.0):
    n_nodes = len(workloads.rsdc_parent_array(branching))
    P = n_nodes - int(np.prod(branching))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    base = torch.randn((B, n_nodes, V + off), generator=gen, device="cuda") * draft_sigma
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    draft = base[:, :P].to(dt)[:, :, off:]
    target = (base + torch.randn((B, n_nodes, V + off), generator=gen, device="cuda")).to(dt)[:, :, off:]
    return draft, target, P


def _tokens(rsd, draft, branching, seed, seq_base=0):
    k, nodes = workloads.rsdc_rows(branching)
    picks = rsd.rsd_gumbel_topk_draft(draft, list(k), list(nodes), seed, 0, seq_base=seq_base)["token"].cpu().numpy()
    return torch.from_numpy(workloads.rsdc_tokens_from_rows(branching, picks)).cuda()


@pytest.mark.parametrize("dtype,V,B,trouble", [("f32", 512, 600, ""), ("bf16", 4096, 600, "nan"), ("bf16", 4104, 600, "far"),
                                               ("f32", 8192, 600, ""), ("bf16", 16392, 150, ""), ("f32", 32768, 150, "nan"),
                                               ("bf16", 65536, 76, ""), ("bf16", 65544, 40, "far"), ("f32", 131072, 40, "")])
def test_cluster_and_ring_walks_give_the_same_bits(dtype, V, B, trouble):
    import paper_2402_14160_b200 as rsd
    branching = (3, 2)
    draft, target, P = _drafted(B, V, dtype, branching, 7000 + V)
    if trouble == "nan":
        draft[::3, 0, V // 2] = float("nan")
        target[1::5, 0, V - 1] = float("nan")
    elif trouble == "far":
        target += 300.0
        draft[::2] -= 120.0
    token = _tokens(rsd, draft, branching, 3)
    parent = torch.from_numpy(workloads.rsdc_parent_array(branching)).cuda()
    whole = rsd.rsd_verify_tree(draft, target, parent, token, 2, 3, 0, want_theta=True)
    n = 5                                                  # a handful of sequences: a cluster each
    for b in (0, B - n):
        part = rsd.rsd_verify_tree(draft[b:b + n], target[b:b + n], parent, token[b:b + n].contiguous(), 2, 3, 0, seq_base=b, want_theta=True)
        for key in part:
            got, want = part[key].cpu().numpy(), whole[key][b:b + n].cpu().numpy()
            assert np.array_equal(got, want, equal_nan=got.dtype.kind == "f"), (key, b)


@pytest.mark.parametrize("dtype,V,B", [("bf16", 511, 9), ("bf16", 4097, 9), ("f32", 8193, 5), ("bf16", 32769, 6), ("f32", 65537, 3),
                                       ("bf16", 131071, 2), ("bf16", 1025, 700)])
@pytest.mark.parametrize("rule,sampler", [(0, 0), (0, 1), (1, 1), (2, 0)])
def test_cluster_walk_off_vector_boundaries_matches_oracle(dtype, V, B, rule, sampler):
    import paper_2402_14160_b200 as rsd
    branching = (2, 3) if V < 60000 else (2, 1)
    draft, target, _ = _drafted(B, V, dtype, branching, 9000 + V, off=1)
    token = _tokens(rsd, draft, branching, 11)
    parent = workloads.rsdc_parent_array(branching)
    g = _np(rsd.rsd_verify_tree_rule(draft, target, torch.from_numpy(parent).cuda(), token, 2, rule, 2.0, sampler, 11, 0, want_theta=True))
    o = oracle.verify_tree(workloads.as_oracle_rows(draft.contiguous()), workloads.as_oracle_rows(target.contiguous()), parent,
                           token.cpu().numpy(), 2, 11, 0, rule=rule, gamma=2.0, final_sampler=sampler)
    t = Tally()
    compare_verify(t, g, o, parent)
    t.check()
    assert np.array_equal(g["status"], o["status"])


@pytest.mark.parametrize("dtype,V", [("f32", 4097), ("bf16", 32768), ("bf16", 131072)])
def test_cluster_residual_draw_with_removed_tokens_in_every_tile_position(dtype, V):
    import paper_2402_14160_b200 as rsd
    B, k = 4, 32                                           # the longest list: first and last token, both sides of tile edges
    _, target, _ = _drafted(B, V, dtype, (1,), 400 + V)
    draft = target[:, 1].clone()
    target = target[:, 0].contiguous()
    edges = [0, 1, 15, 16, 511, 512, 513, V - 1, V - 2, V - 513, 4095, 0]
    rej = np.full((B, k), -1, np.int32)
    for b in range(B):
        rej[b, :] = (edges + [int(x) for x in np.random.RandomState(b).randint(0, V, k - len(edges))])[:k]
    nodes = torch.arange(B, dtype=torch.int32, device="cuda")
    g = _np(rsd.rsd_resample_residual(draft, target, torch.from_numpy(rej).cuda(), nodes, 5, 1, want_residual=True))
    o = oracle.resample_residual(workloads.as_oracle_rows(draft), workloads.as_oracle_rows(target), rej, nodes.cpu().numpy(), 5, 1)
    assert np.all(np.abs(g["residual"] - o["residual"]) <= 1e-5 * o["residual"].max(axis=1, keepdims=True))
    assert np.array_equal(g["status"], o["status"])
    assert np.all(o["margin"][g["token"] != o["token"]] <= 1e-5)

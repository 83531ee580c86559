"""Which kernel walks a sequence is a matter of the batch, the rows and the rule: a cluster that holds the rows on chip (in one of
several shapes), one block or eight that read them in every pass, or, for plain walks over rows on 16-byte boundaries, the ring.
None of it may show: a few sequences alone give the bits they give inside a large batch, and all agree with the oracle."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from tests.launches import launched
from tests.parity import Tally, compare_verify
from tests.test_gpu_parity import _np
from tests.test_gpu_walk_cluster import _drafted, _tokens

pytestmark = pytest.mark.gpu


def _whole_and_parts(rsd, draft, target, parent, token, L, rule=0, gamma=2.0, sampler=0, n=4):
    B = draft.shape[0]
    parent = torch.from_numpy(parent).cuda()
    whole = rsd.rsd_verify_tree_rule(draft, target, parent, token, L, rule, gamma, sampler, 3, 0, want_theta=True)
    for b in (0, B // 2, B - n):
        part = rsd.rsd_verify_tree_rule(draft[b:b + n], target[b:b + n], parent, token[b:b + n].contiguous(), L, rule, gamma, sampler, 3, 0,
                                        seq_base=b, want_theta=True)
        for key in part:
            got, want = part[key].cpu().numpy(), whole[key][b:b + n].cpu().numpy()
            assert np.array_equal(got, want, equal_nan=got.dtype.kind == "f"), (key, b, got, want)
    return whole


# Batches beyond the limits of the on-chip walk, those that four tiles per warp hold, and (rows beyond 131,072 entries) both sides of eight blocks a
# sequence, with the kernel that the whole batch takes; the parts take another, or another shape of it.
@pytest.mark.parametrize("dtype,V,B,off,rule,sampler,trouble,kernel", [
    ("bf16", 32001, 300, 1, 0, 0, "", "walk_stream"), ("bf16", 32001, 230, 7, 0, 0, "nan", "walk_stream"), ("f32", 16389, 600, 3, 0, 0, "nan", "walk_stream"),
    ("bf16", 8201, 800, 1, 0, 0, "far", "walk_stream"), ("bf16", 65551, 200, 1, 0, 0, "far", "walk_stream"), ("bf16", 32000, 300, 0, 1, 0, "", "walk_stream"),
    ("bf16", 16400, 600, 0, 2, 0, "nan", "walk_stream"), ("f32", 8208, 800, 0, 2, 1, "far", "walk_cluster"), ("bf16", 32000, 560, 0, 1, 1, "", "walk_cluster"),
    ("bf16", 32000, 280, 0, 2, 1, "far", "walk_cluster"), ("f32", 8193, 1600, 1, 0, 1, "", "walk_cluster"), ("bf16", 131072, 200, 0, 1, 0, "far", "walk_stream"),
    ("f32", 131073, 240, 1, 0, 0, "nan", "walk_stream"), ("f32", 151936, 240, 0, 0, 0, "far", "walk_stream"), ("bf16", 140001, 160, 1, 2, 0, "", "walk_stream"),
    ("bf16", 262144, 160, 0, 1, 1, "nan", "walk_stream"),
    ("bf16", 32000, 440, 0, 1, 1, "", "walk_stream"), ("bf16", 24001, 440, 1, 2, 1, "far", "walk_stream"), ("f32", 16400, 592, 0, 2, 1, "far", "walk_stream"),
    ("f32", 16401, 592, 1, 0, 1, "nan", "walk_stream"), ("f32", 32004, 290, 0, 2, 0, "", "walk_stream"), ("bf16", 32001, 440, 1, 0, 0, "nan", "walk_stream")])
def test_the_route_of_a_walk_does_not_show(dtype, V, B, off, rule, sampler, trouble, kernel):
    import paper_2402_14160_b200 as rsd
    branching = (3, 2) if B * V < 3e7 else (2, 1)
    draft, target, _ = _drafted(B, V, dtype, branching, 7000 + V, off=off)
    if trouble == "nan":
        draft[::3, 0, V // 2] = float("nan")
        target[1::5, 0, V - 1] = float("nan")
    elif trouble == "far":
        target += 300.0
        draft[::2] -= 120.0
    token = _tokens(rsd, draft, branching, 3)
    parent = workloads.rsdc_parent_array(branching)
    _whole_and_parts(rsd, draft, target, parent, token, 2, rule, 2.0, sampler)
    parent = torch.from_numpy(parent).cuda()
    routes = [launched(lambda: rsd.rsd_verify_tree_rule(draft[:n], target[:n], parent, token[:n], 2, rule, 2.0, sampler, 3, 0)) for n in (B, 4)]
    (whole,), (part,) = routes
    assert whole.kernel == kernel and whole._replace(blocks=0) != part._replace(blocks=0), routes


@pytest.mark.parametrize("dtype,V,B", [("f32", 32000, 400), ("bf16", 32001, 230), ("bf16", 8201, 330), ("f32", 1000, 700), ("f32", 140001, 160), ("bf16", 262144, 310),
                                       ("f32", 16389, 1000), ("bf16", 32001, 440)])
@pytest.mark.parametrize("k", [0, 3])
@pytest.mark.parametrize("trouble", ["", "nan", "far"])
@pytest.mark.parametrize("want_residual", [False, True])
def test_the_route_of_a_residual_draw_does_not_show(dtype, V, B, k, trouble, want_residual):
    import paper_2402_14160_b200 as rsd
    gen = torch.Generator(device="cuda").manual_seed(V + k)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    draft = (torch.randn((B, V), generator=gen, device="cuda") * 2).to(dt)
    target = (draft.float() + torch.randn((B, V), generator=gen, device="cuda")).to(dt)
    if trouble == "nan":
        target[::3, V // 2] = float("nan")
    elif trouble == "far":
        target[::2] += 300.0
        target[:1, 0] = float("nan")
    rejected = torch.randint(0, V, (B, k), generator=gen, device="cuda", dtype=torch.int32) if k else None
    node = torch.arange(B, dtype=torch.int32, device="cuda")
    whole = rsd.rsd_resample_residual(draft, target, rejected, node, 5, 1, want_residual=want_residual)
    n = 3

    def kernel(m):
        return [l._replace(blocks=0) for l in launched(lambda: rsd.rsd_resample_residual(draft[:m], target[:m], rejected[:m] if k else None, node[:m], 5, 1, want_residual=want_residual))]

    # (short rows, and long ones of which nothing is rejected, are drawn from by one kernel whatever the batch)
    assert (kernel(B) != kernel(n)) == (V > 1000 and (k > 0 or V <= 131072))
    for b in (0, B - n):
        for again in (want_residual, not want_residual):          # (asking for the distribution changes the route as well)
            part = rsd.rsd_resample_residual(draft[b:b + n], target[b:b + n], rejected[b:b + n] if k else None, node[b:b + n], 5, 1, seq_base=b,
                                             want_residual=again)
            for key in part:
                if part[key] is not None and whole[key] is not None:
                    assert torch.equal(part[key], whole[key][b:b + n]), (key, b)


@pytest.mark.parametrize("dtype,V,B,off", [("bf16", 140000, 2, 0), ("f32", 140001, 2, 1), ("bf16", 131073, 230, 1), ("f32", 16401, 240, 3), ("bf16", 16401, 300, 1)])
@pytest.mark.parametrize("rule,sampler", [(0, 0), (1, 0), (2, 0), (0, 1), (2, 1)])
def test_walks_over_rows_read_in_every_pass_match_oracle(dtype, V, B, off, rule, sampler):
    import paper_2402_14160_b200 as rsd
    branching = (2, 2) if V * B < 3e5 else (2, 1)
    draft, target, _ = _drafted(B, V, dtype, branching, 9000 + V, off=off)
    token = _tokens(rsd, draft, branching, 11)
    parent = workloads.rsdc_parent_array(branching)
    g = _np(rsd.rsd_verify_tree_rule(draft, target, torch.from_numpy(parent).cuda(), token, 2, rule, 2.0, sampler, 11, 0, want_theta=True))
    n = min(B, 6)                                          # (the rest of a large batch: the test above)
    o = oracle.verify_tree(workloads.as_oracle_rows(draft[:n].contiguous()), workloads.as_oracle_rows(target[:n].contiguous()), parent,
                           token[:n].cpu().numpy(), 2, 11, 0, rule=rule, gamma=2.0, final_sampler=sampler)
    g = {key: v[:n] for key, v in g.items()}
    t = Tally()
    compare_verify(t, g, o, parent)
    t.check()
    assert np.array_equal(g["status"], o["status"])


@pytest.mark.parametrize("dtype,V,B", [("f32", 140001, 3), ("bf16", 262143, 2), ("bf16", 140001, 160), ("f32", 70, 300), ("bf16", 8200, 330)])
@pytest.mark.parametrize("k", [0, 1, 32])
def test_residual_draws_over_rows_read_in_every_pass_match_oracle(dtype, V, B, k):
    import paper_2402_14160_b200 as rsd
    gen = torch.Generator(device="cuda").manual_seed(V + k)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    draft = (torch.randn((B, V), generator=gen, device="cuda") * 2).to(dt)
    target = (draft.float() + torch.randn((B, V), generator=gen, device="cuda")).to(dt)
    rej = None
    k = min(k, V)
    if k:                                                  # both ends of the row and of its tiles, one of them twice; then the draft's favourites
        edges = [V - 1, 0, 511, 512, V - 513, 4096, 0, 1, 15, 16] if V > 5000 else [V - 1, 0, 0, 1, 15, 16]
        rej = np.concatenate([np.tile(np.array(edges[:k], np.int32), (B, 1)),
                              torch.topk(draft.float(), max(1, k - len(edges)), dim=1).indices.int().cpu().numpy()], axis=1)[:, :k].copy()
    nodes = torch.arange(B, dtype=torch.int32, device="cuda")
    g = _np(rsd.rsd_resample_residual(draft, target, None if rej is None else torch.from_numpy(rej).cuda(), nodes, 5, 1, want_residual=True))
    n = min(B, 3)
    o = oracle.resample_residual(workloads.as_oracle_rows(draft[:n]), workloads.as_oracle_rows(target[:n]), None if rej is None else rej[:n],
                                 nodes[:n].cpu().numpy(), 5, 1)
    assert np.all(np.abs(g["residual"][:n] - o["residual"]) <= 1e-5 * o["residual"].max(axis=1, keepdims=True))
    assert np.array_equal(g["status"][:n], o["status"])
    assert np.all(o["margin"][g["token"][:n] != o["token"]] <= 1e-5)


# What large batches seldom meet: the ring (rows on 16-byte boundaries), the streamed walk (off them) and the cluster walk with four tiles per warp against
# small batches, which the oracle tests cover.
@pytest.mark.parametrize("V,B", [(512, 1400), (16389, 260), (16389, 140), (16392, 140)])   # (140 sequences: four tiles per warp; the parts of 40 fewer)
@pytest.mark.parametrize("what", ["repeated", "many_children", "large_tree", "peaked"])
def test_rare_paths_of_large_batches(what, V, B):
    import paper_2402_14160_b200 as rsd
    branching = {"repeated": (4,), "many_children": (32, 2), "large_tree": (20, 20), "peaked": (6, 2)}[what]
    draft, target, P = _drafted(B, V, "bf16", branching, 60 + V)
    if what == "large_tree":
        target = (-1.5 * torch.cat([draft, draft[:, :1].expand(B, target.shape[1] - P, V)], dim=1).float() + 0.3 * target.float()).to(draft.dtype)
    if what == "peaked":                                   # the rejected tokens hold all but a sliver of the draft
        draft[:, :, 7::100] += 18.0
    token = _tokens(rsd, draft, branching, 3)
    if what == "repeated":
        token[:, 3] = token[:, 1]
        target[:, 0].scatter_add_(1, token[:, 1:3].long(), torch.full((B, 2), -9.0, dtype=target.dtype, device="cuda"))
    parent = workloads.rsdc_parent_array(branching)
    if what == "many_children":                            # the last level's 64 nodes become children of the root as well; some repeat
        parent[33:] = 0
        token[::2, 60], token[:, 80], token[::2, 90] = token[::2, 3], token[:, 75], token[::2, 12]
        target[:, 0].scatter_(1, token[:, 1:].long(), -30.0)       # (all of them rejected)
    whole = _whole_and_parts(rsd, draft, target, parent, token, len(branching), n=100 if B != 140 else 40)
    tested = (~torch.isnan(whole["theta"])).sum(dim=1)
    if what == "many_children":
        assert int(tested.min()) >= 96
    if what == "repeated":
        assert int((whole["status"] & rsd.ST_ZERO_DRAFT_PROB != 0).sum()) > B // 2


# A cluster that holds four tiles per warp (the draft's in shared memory) takes the batches that fewer tiles per warp leave waiting: full
# rows of its tiles, one piece more and less, rows off 16-byte boundaries, every rule; against four sequences, which one or two tiles per warp hold.
@pytest.mark.parametrize("dtype,V,B,off,rule,sampler,trouble", [
    ("bf16", 16384, 160, 0, 0, 0, ""), ("bf16", 12288, 290, 0, 1, 1, "nan"), ("bf16", 8193, 200, 1, 0, 0, "far"), ("f32", 32768, 148, 0, 0, 0, "nan"),
    ("bf16", 32760, 100, 0, 0, 0, "far"), ("f32", 16388, 80, 0, 1, 1, ""), ("bf16", 32767, 120, 1, 2, 1, "nan"), ("f32", 32769, 60, 3, 2, 0, "far"),
    ("bf16", 65536, 70, 0, 0, 0, ""), ("bf16", 40008, 60, 0, 2, 1, "nan"), ("f32", 65540, 30, 0, 1, 0, ""), ("bf16", 131072, 33, 0, 0, 0, "nan"),
    ("bf16", 131071, 33, 1, 1, 1, "far"), ("f32", 100001, 24, 1, 0, 1, "nan")])
def test_four_tiles_per_warp_give_the_bits_of_fewer(dtype, V, B, off, rule, sampler, trouble):
    test_the_route_of_a_walk_does_not_show(dtype, V, B, off, rule, sampler, trouble, "walk_stream" if V == 8193 else "walk_cluster")


@pytest.mark.parametrize("dtype,V,B", [("f32", 131072, 33), ("bf16", 65537, 33), ("f32", 32769, 71), ("bf16", 50272, 40)])
@pytest.mark.parametrize("whole", [False, True])
def test_draws_with_nothing_rejected_give_the_same_bits_with_four_tiles_per_warp(dtype, V, B, whole):
    # (one sequence: fewer tiles per warp; the largest batch: the kernel of a block per sequence)
    import paper_2402_14160_b200 as rsd
    gen = torch.Generator(device="cuda").manual_seed(V)
    rows = (torch.randn((4 * B, V), generator=gen, device="cuda") * 2).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    rows[::3, V // 2] = float("nan")
    node = torch.arange(4 * B, dtype=torch.int32, device="cuda")
    all_ = rsd.rsd_resample_residual(rows, rows, None, node, 5, 1, want_residual=whole)
    for b, n in ((0, B), (B - 1, 1), (3 * B, B)):
        part = rsd.rsd_resample_residual(rows[b:b + n], rows[b:b + n], None, node[b:b + n], 5, 1, seq_base=b, want_residual=whole)
        for key in part:
            if part[key] is not None:
                assert torch.equal(part[key], all_[key][b:b + n]), (key, b, n)


@pytest.mark.parametrize("dtype,V,B", [("f32", 16384, 200), ("bf16", 16385, 148), ("f32", 32000, 148), ("bf16", 65529, 64), ("f32", 131072, 33)])
def test_residual_draws_with_four_tiles_per_warp_give_the_bits_of_fewer(dtype, V, B):
    import paper_2402_14160_b200 as rsd
    gen = torch.Generator(device="cuda").manual_seed(V)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    draft = (torch.randn((B, V), generator=gen, device="cuda") * 2).to(dt)
    target = (draft.float() + torch.randn((B, V), generator=gen, device="cuda")).to(dt)
    target[::3, V // 2] = float("nan")
    rejected = torch.randint(0, V, (B, 32), generator=gen, device="cuda", dtype=torch.int32)
    edges = [0, 511, 512, V - 1, V - 512, 0, 15, 16384 % V, 8191, 8192]        # both ends of tiles, of a warp's share and of the row; one of them twice
    rejected[:, : len(edges)] = torch.tensor(edges, dtype=torch.int32, device="cuda")
    node = torch.arange(B, dtype=torch.int32, device="cuda")
    whole = rsd.rsd_resample_residual(draft, target, rejected, node, 5, 1, want_residual=True)
    for b in (0, B - 3):
        part = rsd.rsd_resample_residual(draft[b:b + 3], target[b:b + 3], rejected[b:b + 3], node[b:b + 3], 5, 1, seq_base=b, want_residual=True)
        for key in part:
            assert torch.equal(part[key], whole[key][b:b + 3]), (key, b)


# Where the two costs of a walk that four tiles per warp could hold lie clearly apart (us, on chip / the other route): the faster one is taken.
@pytest.mark.parametrize("dtype,V,B,off,rule,expected", [
    ("f32", 130695, 101, 0, 0, "walk_cluster"),            # (3, 2) tree: about 150 / 296
    ("f32", 46630, 79, 0, 0, "walk_cluster"),              # 57 / 98
    ("f32", 65840, 59, 1, 0, "walk_cluster"),              # 62 / 101
    ("f32", 118688, 102, 1, 0, "walk_cluster"),            # 184 / 289
    ("bf16", 110439, 180, 0, 2, "walk_stream"), ("bf16", 32000, 148, 0, 0, "walk_cluster"), ("bf16", 32000, 444, 0, 0, "verify_tree_ring"),
    ("f32", 16389, 900, 3, 0, "walk_stream"), ("bf16", 131073, 4, 0, 0, "walk_stream"), ("bf16", 262144, 4, 0, 0, "verify_tree_ring")])
def test_walks_take_the_faster_route(dtype, V, B, off, rule, expected):
    import paper_2402_14160_b200 as rsd
    draft, target, _ = _drafted(B, V, dtype, (2, 1), 5, off=off)
    token = _tokens(rsd, draft, (2, 1), 3)
    parent = torch.from_numpy(workloads.rsdc_parent_array((2, 1))).cuda()
    assert [l.kernel for l in launched(lambda: rsd.rsd_verify_tree_rule(draft, target, parent, token, 2, rule, 2.0, 0, 3, 0))] == [expected]


def _draw_launches(dtype, V, B, k, whole):
    import paper_2402_14160_b200 as rsd
    rows = torch.randn((B, V), device="cuda").to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    rejected = torch.randint(0, V, (B, k), device="cuda", dtype=torch.int32) if k else None
    node = torch.zeros(B, dtype=torch.int32, device="cuda")
    return launched(lambda: rsd.rsd_resample_residual(rows, rows, rejected, node, 5, 1, want_residual=whole))


@pytest.mark.parametrize("dtype,V,B,k,whole,expected", [
    ("bf16", 104256, 106, 1, False, "walk_stream"),        # 67 / 52
    ("f32", 48448, 216, 1, False, "walk_stream"),          # 52 / 40
    ("bf16", 31296, 285, 1, False, "walk_stream"),         # 41 / 31
    ("f32", 110336, 207, 1, False, "walk_stream"),         # 101 / 79
    ("bf16", 90624, 16, 0, True, "walk_cluster"), ("f32", 69744, 18, 0, False, "walk_cluster"), ("f32", 50591, 34, 0, True, "walk_cluster"),   # 13 / 36, 9 / 19, 17 / 29
    ("bf16", 122904, 34, 0, False, "draw_target"), ("bf16", 60000, 34, 0, False, "draw_target"), ("bf16", 32000, 148, 0, True, "draw_target"),
    ("bf16", 104256, 106, 16, False, "walk_cluster"), ("f32", 32000, 256, 3, True, "walk_cluster"), ("bf16", 8000, 900, 3, True, "walk_cluster")])
def test_residual_draws_take_the_faster_route(dtype, V, B, k, whole, expected):
    assert [l.kernel for l in _draw_launches(dtype, V, B, k, whole)] == [expected]

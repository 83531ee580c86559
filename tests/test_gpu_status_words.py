"""The status words of the drafting and filtering calls are cleared by a kernel of 256-thread blocks that the next kernel
overlaps: whatever the words held, afterwards they hold this call's bits and nothing else, at the edges of a block."""
import pytest
import torch

from tests.launches import launched

pytestmark = pytest.mark.gpu
NAN_INPUT = 1


@pytest.mark.parametrize("B", [1, 255, 256, 257, 513])
@pytest.mark.parametrize("call", ["draft", "filter"])
def test_status_words_hold_the_bits_of_their_own_call(call, B):
    import paper_2402_14160_b200 as rsd
    clean = torch.randn((B, 2, 640), generator=torch.Generator(device="cuda").manual_seed(B), device="cuda")
    marked = clean.clone()
    marked[::3, 1, 600] = float("nan")
    marked[B - 1, 0, 3] = float("nan")

    def run(rows, out=None):
        if call == "draft":
            return rsd.rsd_gumbel_topk_draft(rows, [2, 2], [0, 1], 7, 1, out=out)
        return rsd.rsd_filter_rows(rows, 20, 0.9, out=out)

    want = torch.isnan(marked).any(dim=2).any(dim=1).to(torch.int32) * NAN_INPUT
    out = run(clean)
    out["status"].fill_(-1)
    got = []
    for rows in (marked, clean, marked, clean):          # one behind the other, into the same words
        run(rows, out)
        got.append(out["status"].clone())
    for g, w in zip(got, (want, want * 0, want, want * 0)):
        assert torch.equal(g, w)


@pytest.mark.parametrize("B", [1, 3, 300])
def test_status_of_sequences_of_one_row_is_stored(B):
    # no kernel ahead clears it: every sequence's word is written, whatever it held
    import paper_2402_14160_b200 as rsd
    rows = torch.randn((B, 1, 9000), device="cuda")
    rows[::2, 0, 5] = float("nan")
    out = rsd.rsd_filter_rows(rows, 0, 0.9)
    out["status"].fill_(77)
    rsd.rsd_filter_rows(rows, 0, 0.9, out=out)
    assert out["status"].cpu().tolist() == [rsd.ST_NAN_INPUT if b % 2 == 0 else 0 for b in range(B)]


@pytest.mark.parametrize("B,R,V", [(1, 1, 20000), (1, 7, 32000), (3, 8, 5000), (3, 9, 5000), (46, 8, 17000), (47, 8, 17000), (2, 8, 70000)])
def test_status_of_few_rows_gathered_by_their_cluster(B, R, V):
    # up to eight rows a sequence, few in all: a cluster's first block stores the OR of their bits; the other sizes clear and OR
    import paper_2402_14160_b200 as rsd
    rows = torch.randn((B, R, V), device="cuda")
    want = [0] * B
    rows[0, R - 1, V - 1] = float("nan")
    want[0] |= NAN_INPUT
    if B > 1:
        rows[B - 1, 0, 2:] = float("-inf")               # fewer entries than picks
        want[B - 1] |= rsd.ST_FEWER_THAN_K
        rows[B - 1, R - 1, 7] = float("nan")
        want[B - 1] |= NAN_INPUT
    for values in (False, True):
        out = rsd.rsd_gumbel_topk_draft(rows, [3] * R, list(range(R)), 1, 0, want_values=values)
        out["status"].fill_(77)
        rsd.rsd_gumbel_topk_draft(rows, [3] * R, list(range(R)), 1, 0, want_values=values, out=out)
        assert out["status"].cpu().tolist() == want


# Close to one row an SM (148) the blocks of a cluster share SMs: 4-byte rows off 32-byte boundaries with 512 threads have their words cleared.
@pytest.mark.parametrize("dtype,B,R,V,clusters", [
    ("f32", 16, 7, 58589, False), ("f32", 34, 4, 36910, False), ("f32", 11, 8, 20001, True), ("f32", 30, 5, 20001, True), ("f32", 140, 1, 20001, True),
    ("f32", 16, 7, 32000, True), ("bf16", 16, 7, 58589, True), ("f32", 12, 9, 20001, False)])
def test_rows_that_would_share_an_sm_as_clusters_have_their_words_cleared(dtype, B, R, V, clusters):
    import paper_2402_14160_b200 as rsd
    rows = torch.randn((B, R, V), device="cuda").to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    rows[::2, R - 1, V - 1] = float("nan")
    out = rsd.rsd_gumbel_topk_draft(rows, [3] * R, list(range(R)), 1, 0)
    out["status"].fill_(77)
    got = launched(lambda: rsd.rsd_gumbel_topk_draft(rows, [3] * R, list(range(R)), 1, 0, out=out))
    assert [l.kernel for l in got] == (["scan_topk"] if clusters else ["clear_status", "scan_topk"])
    assert got[-1].cluster == (R if clusters else 0)
    assert out["status"].cpu().tolist() == [NAN_INPUT if b % 2 == 0 else 0 for b in range(B)]


# Lone rows: launches of rows beyond 4096 entries that come close to one or two an SM (148) start in plain stream order, the others overlap the end of
# what is ahead.
@pytest.mark.parametrize("B", [74, 75, 148, 149, 222, 223, 296, 297])
@pytest.mark.parametrize("V", [4096, 9001])
def test_filter_calls_behind_each_other_read_what_the_one_before_wrote(B, V):
    import paper_2402_14160_b200 as rsd
    rows = torch.randn((B, 1, V), device="cuda")
    rows[::2, 0, 5] = float("nan")
    outs = [rsd.rsd_filter_rows(rows, 0, 1.0) for _ in range(4)]
    torch.cuda.synchronize()

    def chain(wait):
        src = rows
        for out in outs:
            out["status"].fill_(77)
            out["rows"].fill_(1.0)
        for i, (top_k, top_p) in enumerate(((3000, 0.99), (700, 0.95), (90, 0.9), (0, 0.5))):
            if wait:
                torch.cuda.synchronize()
            rsd.rsd_filter_rows(src, top_k, top_p, out=outs[i])
            src = outs[i]["rows"]
        return [{k: v.clone() for k, v in o.items()} for o in outs]

    for got, want in zip(chain(False), chain(True)):
        for key in got:
            assert torch.equal(got[key], want[key]), key
    assert outs[0]["status"].cpu().tolist() == [NAN_INPUT if b % 2 == 0 else 0 for b in range(B)]
    assert not bool(outs[3]["status"].any())

"""rsd_sbs_draft_tree keeps a sequence's finalists, and their noise, in shared memory as far as they fit: at the tree sizes
where either stops fitting the results stay those of one rsd_sbs_step call per level, bit for bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,L", [(8, 29), (8, 30), (11, 15), (11, 16), (11, 24), (12, 20), (16, 11),
                                 (16, 12), (24, 4), (32, 2)])
@pytest.mark.parametrize("is_logprob", [False, True])
def test_wide_trees_are_the_chain_of_level_calls(W, L, is_logprob):
    import paper_2402_14160_b200 as rsd
    B, V = 3, 600
    P = 1 + (L - 1) * W
    draft = torch.randn((B, P, V), generator=torch.Generator(device="cuda").manual_seed(10 * W + L), device="cuda") * 2
    if is_logprob:
        draft = torch.log_softmax(draft, -1)
    token, parent = (torch.full((B, 1 + L * W), -1, dtype=torch.int32, device="cuda") for _ in range(2))
    whole = rsd.rsd_sbs_draft_tree(draft, W, L, 5, 1, token, parent, is_logprob=is_logprob)
    prev = None
    for l in range(L):
        first, n_par = (0, 1) if l == 0 else (1 + (l - 1) * W, W)
        prev = rsd.rsd_sbs_step(draft[:, first:first + n_par], W, first, prev and prev["sum_logprob"], prev and prev["trunc_gumbel"], 5, 1,
                                is_logprob=is_logprob, parent_base=first)
        nodes = slice(1 + l * W, 1 + (l + 1) * W)
        assert torch.equal(token[:, nodes], prev["token"]) and torch.equal(parent[:, nodes], prev["parent"]), l
        assert torch.equal(whole["count"][l], prev["count"])
    assert torch.equal(whole["sum_logprob"], prev["sum_logprob"]) and torch.equal(whole["trunc_gumbel"], prev["trunc_gumbel"])

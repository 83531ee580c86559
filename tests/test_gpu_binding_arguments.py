"""The binding refuses what is not an integer where an integer is due (seed, step, sequence base, node numbers) instead of
cutting it, and converts where int() or float() always stood (sizes of a filter, rules, temperatures)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _calls(rsd, api):
    B, V = 2, 64
    rows = torch.randn((B, 3, V), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    parent = torch.tensor([-1, 0, 0], dtype=torch.int32, device="cuda")
    token = torch.tensor([[-1, 3, 5]] * B, dtype=torch.int32, device="cuda")
    node = torch.zeros((B,), dtype=torch.int32, device="cuda")
    tree = torch.full((B, 5), -1, dtype=torch.int32, device="cuda")
    level = dict(token=tree[:, 1:3], parent=tree[:, 3:5], sum_logprob=torch.empty((B, 2), device="cuda"),
                 trunc_gumbel=torch.empty((B, 2), device="cuda"), count=node.clone(), status=node.clone())
    return {
        "draft": lambda seed=1, step=2, seq_base=3: rsd.rsd_gumbel_topk_draft(rows, [1, 1, 2], [0, 1, 2], seed, step, seq_base=seq_base),
        "level": lambda seed=1, step=2, seq_base=3, first=0, base=0: api.rsd_sbs_step_static(rows[:, :1], 2, first, None, None, seed, step, level, seq_base=seq_base,
                                                                                             parent_base=base),
        "tree": lambda seed=1, step=2, seq_base=3: rsd.rsd_sbs_draft_tree(rows, 2, 2, seed, step, tree, tree.clone(), seq_base=seq_base),
        "walk": lambda seed=1, step=2, seq_base=3: rsd.rsd_verify_tree(rows[:, :1], rows, parent, token, 1, seed, step, seq_base=seq_base),
        "residual": lambda seed=1, step=2, seq_base=3: rsd.rsd_resample_residual(rows[:, 0], rows[:, 1], None, node, seed, step, seq_base=seq_base),
    }


@pytest.mark.parametrize("bad", [1.5, 2.0, "3", None])
def test_what_is_not_an_integer_is_refused(bad):
    import paper_2402_14160_b200 as rsd
    from paper_2402_14160_b200 import api
    for name, call in _calls(rsd, api).items():
        call()
        for arg in ("seed", "step", "seq_base") + (("first", "base") if name == "level" else ()):
            with pytest.raises(TypeError):
                call(**{arg: bad})


def test_what_int_and_float_take_is_taken():
    import paper_2402_14160_b200 as rsd
    rows = torch.randn((2, 1, 64), generator=torch.Generator(device="cuda").manual_seed(2), device="cuda")
    want = rsd.rsd_filter_rows(rows, 5, 0.5, temperature=0.75)["rows"]
    for top_k, top_p, T in ((5.0, "0.5", np.float32(0.75)), (np.int64(5), np.float64(0.5), torch.tensor(0.75))):
        assert torch.equal(rsd.rsd_filter_rows(rows, top_k, top_p, temperature=T)["rows"], want)
    with pytest.raises((TypeError, ValueError)):
        rsd.rsd_filter_rows(rows, 5, "a half")

"""The row scan uses 128, 256 or 512 threads per row, by the number of rows and their length, and reads rows off 32-byte
boundaries in shifted words.  None of this may show: a few rows scanned alone give the bits they give inside a large
batch (picks, perturbed values and log-probabilities), at the sizes where the number of threads changes.

With a log-sum-exp (the first test) that is 128 threads against 256 with the sums on four warps, from 16,384 to 65,536 entries;
its other sizes run one kernel whatever the batch and are there for the oracle and the shifted words.  Without one (the second
test: picks only, or rows of log-probabilities) it is all three."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from tests.launches import launched
from tests.parity import Tally, compare_topk

pytestmark = pytest.mark.gpu


def _draft(rows, k, seq_base, is_logprob=False, temperature=1.0):
    import paper_2402_14160_b200 as rsd
    out = rsd.rsd_gumbel_topk_draft(rows, [k], [2], 17, 3, seq_base=seq_base, want_values=True, is_logprob=is_logprob, temperature=temperature)
    return {key: v.cpu().numpy() for key, v in out.items()}


@pytest.mark.parametrize("dtype,V,B,off,trouble", [
    ("bf16", 4096, 700, 0, ""), ("f32", 4080, 300, 0, "jump"), ("bf16", 16384, 500, 0, "jump"), ("f32", 32000, 400, 0, "nan"), ("bf16", 32016, 400, 8, ""),
    ("bf16", 32001, 400, 0, "nan"), ("f32", 16389, 400, 3, "jump"), ("bf16", 65552, 300, 0, ""), ("f32", 131072, 240, 0, ""),
    ("bf16", 65537, 300, 1, "")])
def test_rows_alone_and_in_a_batch_give_the_same_bits(dtype, V, B, off, trouble):
    gen = torch.Generator(device="cuda").manual_seed(V + B)
    rows = torch.randn((B, 1, V + off), generator=gen, device="cuda") * 2
    if trouble == "jump":        # maxima that jump by more than the log-sum-exp's reference allows, and chunks of -inf
        rows[::2, :, V // 2::97] += 60.0
        rows[1::3, :, :3000] = float("-inf")
    elif trouble == "nan":
        rows[::4, :, V - 1 + off] = float("nan")
    rows = rows.to(torch.bfloat16 if dtype == "bf16" else torch.float32)[:, :, off:]
    whole = _draft(rows, 8, 5)
    for b, n in ((0, 3), (B - 2, 2), (B // 2, 160)):
        n = min(n, B - b)
        part = _draft(rows[b:b + n], 8, 5 + b)
        for key in part:
            assert np.array_equal(part[key], whole[key][b:b + n], equal_nan=part[key].dtype.kind == "f"), (key, b)
    n = 2
    o = oracle.gumbel_topk(workloads.as_oracle_rows(rows[:n].contiguous()), [8], [2], 17, 3, seq_base=5)
    t = Tally()
    # an fp32 log-probability is a difference of terms of up to 70: two ulps of that on top of the usual 1e-6
    compare_topk(t, whole["token"][:n], o, [8], whole["perturbed"][:n], whole["logprob"][:n], logprob_abs_tol=1e-6 + 2 * 70 * 1.2e-7)
    t.check()


# rows on both sides of 1.5 and 2.5 per SM (222 and 370 of 148): 128 / 256 threads from 4096 entries, 128 / 256 / 512 from 16,384,
# 2-byte rows of more than 65,536 entries 256 / 512, 4-byte ones always 512
@pytest.mark.parametrize("dtype,V,B,off,trouble", [
    ("bf16", 4096, 380, 0, ""), ("f32", 4111, 240, 1, "nan"), ("bf16", 16383, 380, 3, "jump"), ("f32", 16384, 380, 0, "jump"), ("bf16", 32001, 380, 0, "nan"),
    ("f32", 32000, 380, 0, ""), ("bf16", 65552, 300, 0, "jump"), ("bf16", 65537, 300, 1, ""), ("f32", 65552, 60, 0, "nan")])
@pytest.mark.parametrize("form", ["picks", "logprob", "tempered picks"])
def test_rows_without_log_sum_exp_alone_and_in_a_batch_give_the_same_bits(dtype, V, B, off, trouble, form):
    import paper_2402_14160_b200 as rsd
    gen = torch.Generator(device="cuda").manual_seed(3 * V + B)
    rows = torch.randn((B, 1, V + off), generator=gen, device="cuda") * 2
    if form == "logprob":
        rows = torch.log_softmax(rows, -1)
    if trouble == "jump":
        rows[::2, :, V // 2::97] += 20.0
        rows[1::3, :, :3000] = float("-inf")
    elif trouble == "nan":
        rows[::4, :, V - 1 + off] = float("nan")
    rows = rows.to(torch.bfloat16 if dtype == "bf16" else torch.float32)[:, :, off:]
    T = 0.3 if form == "tempered picks" else 1.0

    def scan(part, seq_base):
        out = rsd.rsd_gumbel_topk_draft(part, [8], [2], 17, 3, seq_base=seq_base, is_logprob=form == "logprob", want_values=form == "logprob", temperature=T)
        return {key: v.cpu().numpy() for key, v in out.items() if v is not None}

    whole = scan(rows, 5)
    for b, n in ((0, 3), (B - 2, 2), (B // 4, 150), (10, 230)):
        n = min(n, B - b)
        part = scan(rows[b:b + n], 5 + b)
        for key in part:
            assert np.array_equal(part[key], whole[key][b:b + n], equal_nan=part[key].dtype.kind == "f"), (key, b)
    n = 2
    o = oracle.gumbel_topk(workloads.as_oracle_rows(rows[:n].contiguous()), [8], [2], 17, 3, seq_base=5, is_logprob=form == "logprob", temperature=T)
    t = Tally()
    compare_topk(t, whole["token"][:n], o, [8], *([whole["perturbed"][:n], whole["logprob"][:n]] if form == "logprob" else []))
    t.check()


# A level of few rows runs in one launch (the rows of a sequence as a cluster, 128 to 512 threads a row), one of many rows in two.
@pytest.mark.parametrize("dtype,V,n_par,W,B,off,form,trouble", [
    ("bf16", 70, 8, 8, 200, 0, "", "few"), ("f32", 4096, 3, 5, 200, 0, "", "nan"), ("bf16", 16383, 8, 32, 60, 1, "tempered", ""), ("f32", 16384, 2, 2, 300, 0, "", "dead"),
    ("bf16", 32000, 4, 4, 140, 0, "", "nan"), ("f32", 32000, 6, 6, 80, 0, "logprob", "dead"), ("f32", 1001, 7, 3, 90, 1, "logprob", "few"),
    ("bf16", 65552, 8, 8, 64, 0, "", "dead"), ("f32", 70001, 5, 8, 90, 3, "tempered", "nan"), ("bf16", 131072, 1, 8, 400, 0, "", ""),
    ("bf16", 2047, 8, 32, 60, 1, "tempered", ""), ("bf16", 40001, 8, 16, 60, 1, "", "nan"), ("f32", 58816, 2, 2, 99, 0, "", "dead"), ("f32", 58589, 7, 7, 16, 3, "logprob", "nan")])
def test_levels_alone_and_in_a_batch_give_the_same_bits(dtype, V, n_par, W, B, off, form, trouble):
    import paper_2402_14160_b200 as rsd
    gen = torch.Generator(device="cuda").manual_seed(V + B)
    rows = torch.randn((B, n_par, V + off), generator=gen, device="cuda") * 2
    if form == "logprob":
        rows = torch.log_softmax(rows, -1)
    if trouble == "nan":
        rows[::4, n_par - 1, V - 1 + off] = float("nan")
    elif trouble == "few":       # fewer entries than children
        rows[::2, :, off + 2:] = float("-inf")
    rows = rows.to(torch.bfloat16 if dtype == "bf16" else torch.float32)[:, :, off:]
    total = -torch.rand((B, n_par), generator=gen, device="cuda")
    gumbel = torch.randn((B, n_par), generator=gen, device="cuda")
    if trouble == "dead":        # parent slots that the level above left empty
        total[::3, n_par - 1] = gumbel[::3, n_par - 1] = float("-inf")
    T = 0.4 if form == "tempered" else 1.0

    def level(b, n):
        sums = (None, None) if n_par == 1 else (total[b:b + n].contiguous(), gumbel[b:b + n].contiguous())
        return rsd.rsd_sbs_step(rows[b:b + n], W, 3, *sums, 17, 3, is_logprob=form == "logprob", seq_base=5 + b, temperature=T)

    whole = level(0, B)
    for b, n in ((0, 1), (B // 2, 3), (B - 2, 2)):
        part = level(b, n)
        for key in part:
            got, want = part[key].cpu().numpy(), whole[key][b:b + n].cpu().numpy()
            assert np.array_equal(got, want, equal_nan=got.dtype.kind == "f"), (key, b)


# Up to 16 children of longer rows; 4-byte rows with a log-sum-exp up to half as many as SMs from 48,000 to 65,536 entries, beyond that only whole groups.
@pytest.mark.parametrize("dtype,V,n_par,W,B,logprob,one", [
    ("bf16", 32000, 4, 16, 8, False, True), ("bf16", 32000, 4, 17, 8, False, False), ("bf16", 2048, 4, 32, 8, False, True), ("bf16", 2049, 4, 32, 8, False, False),
    ("f32", 58816, 2, 2, 99, False, False), ("f32", 58816, 2, 2, 37, False, True), ("f32", 48000, 2, 2, 99, False, True), ("f32", 58816, 2, 2, 99, True, True),
    ("f32", 70001, 5, 5, 10, False, False), ("f32", 70000, 5, 5, 10, False, True), ("f32", 58589, 7, 7, 16, True, False), ("f32", 58592, 7, 7, 16, True, True),
    ("bf16", 65535, 6, 6, 24, False, True), ("bf16", 32000, 9, 8, 2, False, False)])
def test_levels_take_the_faster_route(dtype, V, n_par, W, B, logprob, one):
    import paper_2402_14160_b200 as rsd
    rows = torch.randn((B, n_par, V), device="cuda")
    rows = (torch.log_softmax(rows, -1) if logprob else rows).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    sums = torch.zeros((B, n_par), device="cuda")
    got = launched(lambda: rsd.rsd_sbs_step(rows, W, 3, sums, sums, 17, 3, is_logprob=logprob))
    assert [l.kernel for l in got] == (["scan_level"] if one else ["scan_topk", "sbs_epilogue"])

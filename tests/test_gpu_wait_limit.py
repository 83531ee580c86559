"""A walk whose wait for another block's sums runs out reports it: every output of its sequence is written and the status says
RSD_ST_TIMEOUT, whichever block of the cluster gave up.

A variant of the library whose waits run out unless the words are there already (-DRSD_WAIT_CYCLES=-1) is run in a child
process (the binding loads one library per process), on batches that clusters walk; a sequence without the bit must hold what
the ordinary library gives."""
import os
import subprocess
import sys
import tempfile

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys
sys.path.insert(0, %(root)r)
import torch
import workloads
import paper_2402_14160_b200 as rsd
from paper_2402_14160_b200 import api


def untouched(shape, dtype, device):     # a word that no call writes by itself
    return torch.full((shape,) if isinstance(shape, int) else tuple(shape), 77, dtype=dtype, device=device)


api._new = untouched
out = {}
for V, dtype, B in [(512, torch.float32, 40), (32000, torch.bfloat16, 24), (32001, torch.float32, 9), (131072, torch.bfloat16, 6)]:
    branching = (3, 2)
    parent = workloads.rsdc_parent_array(branching)
    g = torch.Generator(device="cuda").manual_seed(V)
    target = (torch.randn((B, len(parent), V), generator=g, device="cuda") * 2).to(dtype)
    draft = (target[:, :4] + torch.randn((B, 4, V), generator=g, device="cuda")).to(dtype)
    token = torch.randint(0, V, (B, len(parent)), generator=g, device="cuda", dtype=torch.int32)
    par = torch.from_numpy(parent).cuda()
    for rule, sampler in [(0, 0), (1, 1), (2, 0)]:
        r = rsd.rsd_verify_tree_rule(draft, target, par, token, 2, rule, 2.0, sampler, 3, 0)
        out[(V, rule)] = {k: v.cpu() for k, v in r.items() if v is not None}
    r = rsd.rsd_resample_residual(draft[:, 0].contiguous(), target[:, 0].contiguous(), token[:, 1:4].contiguous(),
                                  torch.arange(B, dtype=torch.int32, device="cuda"), 3, 0, want_residual=True)
    out[(V, "residual")] = {k: v.cpu() for k, v in r.items() if k != "residual"}
torch.save(out, sys.argv[1])
"""


def test_a_wait_that_runs_out_is_reported_whichever_block_gave_up():
    import torch
    from paper_2402_14160_b200 import build, api
    TIMEOUT = api.ST_TIMEOUT
    got = []
    with tempfile.TemporaryDirectory() as d:
        impatient = build.build(out=os.path.join(d, "librsd_impatient.so"), defines=("RSD_WAIT_CYCLES=-1",))
        for lib in (impatient, build.LIB):
            path = os.path.join(d, "out.pt")
            r = subprocess.run([sys.executable, "-c", CHILD % {"root": ROOT}, path], env=dict(os.environ, RSD_LIB_PATH=lib),
                               capture_output=True, text=True, timeout=600)
            assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
            got.append(torch.load(path))
    given_up = 0
    for key, want in got[1].items():
        assert not (want["status"] & TIMEOUT).any()
        for b in range(len(want["status"])):
            have = {name: t[b] for name, t in got[0][key].items()}
            last = have["token"] if "token" in have else have["last_token"]
            if have["status"] & TIMEOUT:
                given_up += 1
                assert have["status"] < 64 and last == -1, (key, b, have)
                if "accepted_len" in have:
                    n = int(have["accepted_len"])
                    assert 0 <= n <= 2 and 0 <= have["stop_reason"] <= 2, (key, b, have)
                    assert (have["accepted_node"][:n] > 0).all() and (have["accepted_node"][n:] == -1).all(), (key, b, have)
            else:
                assert all(torch.equal(have[name], want[name][b]) for name in have), (key, b, have)
    assert given_up > 0

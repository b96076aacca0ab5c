"""sva_attend_nodes_noalloc, the attention entry point for callers that may
not allocate device memory (for example a plugin whose host framework gives
it only its input and output buffers): the library takes the key-range split
scratch from its own static device array instead of a caller workspace.

Through the C ABI, on two calls in a row, its output must match what
sva_attend_nodes with a workspace computes on the same inputs, within the
tolerances of the other parity tests (and, since both take the same split
plan, bit for bit); on clean1 it is also checked against the oracle.  A
launch whose wave-filling split needs more scratch than the array holds must
be refused without launching anything.  That split, by which the limit is
stated, is worked out here from the device's SM count (full waves unsplit, the
partial last wave split); the plan that a launch takes also counts what a
merge costs and may merge inside clusters or not split at all.  This file runs last so that a failure here cannot
hide the results of the other tests, and it depends on no state they leave
behind."""
import ctypes
import subprocess
import sys

import numpy as np
import pytest
import torch

from paper_2609_22283_gb300 import inputs as I
from paper_2609_22283_gb300 import sva
from paper_2609_22283_gb300.pipeline import Step
from tests import _parity as P
from tests.conftest import ROOT

pytestmark = pytest.mark.gpu

MAX_ABS = P.MAX_ABS   # element bound 2e-2 + ulp_bf16(|O|) / 2, as in the parity tests
REL_RMS = P.REL_RMS
STATIC_SCRATCH = 32 << 20
MAX_SPLIT = 4

# 1 node, 2 heads x 128, T = 240, clean history of 7 chunks: 2 work units of
# 16 key tiles each, whose wave-filling split is 4 ways (about 1 MB of scratch)
# and which are merged inside clusters.
SPLIT4 = I.Workload(name="split4", seed=9, F=1, Hp=8, Wp=30, H=2, d=128, K=4, W=7,
                    policy="clean", nodes=((0, 9, 4),),
                    prefilled=tuple((0, c, 0) for c in range(2, 9)))

# 8 sequences of the same, 20 heads: 160 work units, one wave of 152 unsplit and
# 8 split 4 ways, merged through the scratch.
MERGE4 = I.Workload(name="merge4", seed=10, F=1, Hp=8, Wp=30, H=20, d=128, K=4, W=7,
                    policy="clean", nodes=tuple((s, 9, 4) for s in range(8)),
                    prefilled=tuple((s, c, 0) for s in range(8) for c in range(2, 9)))


def _plan(units, min_tiles, sms, cap):
    """(n_full, n_split) of the wave-filling split: the number of splits
    minimising waves per split, the full waves unsplit when that is no worse."""
    def choose(u):
        best, best_s = float(-(-u // sms)), 1
        for s in range(2, MAX_SPLIT + 1):
            if u * s > cap or min_tiles // s < 4:
                break
            cost = -(-(u * s) // sms) / s
            if cost < best - 1e-9:
                best, best_s = cost, s
        return best_s
    s_all = choose(units)
    if units < sms:
        return 0, s_all
    full = units // sms * sms
    rest = units - full
    s_rest = choose(rest)
    cost_all = -(-(units * s_all) // sms) / s_all
    cost_mixed = full / sms + -(-(rest * s_rest) // sms) / s_rest
    return (full, s_rest) if cost_mixed <= cost_all + 1e-9 else (0, s_all)


def _scratch(w, sms):
    """(n_split, bytes of scratch) of the wave-filling split of a dense launch of workload w."""
    nt = w.tiles
    units = w.H * w.n_nodes * -(-nt // 2)
    min_tiles = min((1 + max(0, min(w.W, b - 1))) * nt for (_, b, _) in w.nodes)
    n_full, n_split = _plan(units, min_tiles, sms, 4 * sms)
    if n_split == 1:
        return 1, 0
    split_units = units - n_full
    return n_split, (-(-split_units * 4 // 256) * 256) + split_units * n_split * 256 * (w.d + 2) * 4


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _noalloc(step, nodes, q, out, lse):
    lib = sva.load()
    return lib.sva_attend_nodes_noalloc(
        step.cache.handle, nodes, len(nodes), ctypes.c_void_p(q.data_ptr()),
        ctypes.c_void_p(out.data_ptr()), ctypes.c_void_p(lse.data_ptr() if lse is not None else 0),
        step.scale, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))


@pytest.mark.parametrize("name", ["split4", "merge4", "tiny", "clean1"])
def test_noalloc_matches_attend_nodes_twice(name):
    w = {"split4": SPLIT4, "merge4": MERGE4}.get(name) or I.WORKLOADS[name]
    n_split, need = _scratch(w, _sms())
    if name != "tiny":
        assert n_split > 1 and 0 < need <= STATIC_SCRATCH, (n_split, need)
    inp = I.generate(w)
    step = Step(w, workspace=True)
    step.prefill(inp)
    q, k, v = step.device_inputs(inp)
    ref, ref_lse = step.outputs()
    step.run(q, k, v, ref, ref_lse)                 # sva_attend_nodes, caller workspace
    assert step.cache.poll() == sva.OK
    nodes, _ = step.node_table()
    b = ref.float()
    for call in range(2):
        out = torch.full_like(ref, float("nan"))
        lse = torch.full_like(ref_lse, float("nan"))
        assert _noalloc(step, nodes, q, out, lse) == sva.OK, sva.last_error()
        assert step.cache.poll() == sva.OK
        a = out.float()
        assert torch.isfinite(a).all(), f"call {call}: unwritten output"
        bound = MAX_ABS + 0.5 * torch.from_numpy(P.ulp_bf16(b.cpu().numpy())).to(b.device)
        assert bool(((a - b).abs() <= bound).all()), call
        rel = (torch.linalg.norm(a - b) / torch.linalg.norm(b)).item()
        assert rel <= REL_RMS, (call, rel)
        np.testing.assert_allclose(lse.cpu().numpy(), ref_lse.cpu().numpy(), atol=2e-3, rtol=0)
        # the same split plan and kernel: the same bits
        assert torch.equal(out.view(torch.int16), ref.view(torch.int16)), call
    if name == "clean1":
        got = out.cpu()
        states = P.oracle_states(w, inp)
        rows = I.sample_rows(w, 64, seed=17)
        oref, _ = P.oracle_node(w, inp, states, 0, range(w.H), rows)
        for h in range(w.H):
            P.assert_close(got[0, rows, h, :].float().numpy(), oref[h], f"noalloc clean1 head {h}")
    step.close()


def test_noalloc_refuses_plan_beyond_its_scratch():
    # One node of 240 tokens (one work unit per head, 16 key tiles) over 7
    # clean history chunks; the head count is the smallest whose wave-filling
    # split on this GPU needs more than the static scratch.
    sms = _sms()
    w = None
    for H in range(1, 129):
        cand = I.Workload(name="wide", seed=12, F=1, Hp=8, Wp=30, H=H, d=128, K=4, W=7,
                          policy="clean", nodes=((0, 9, 4),),
                          prefilled=tuple((0, c, 0) for c in range(2, 9)))
        if _scratch(cand, sms)[1] > STATIC_SCRATCH:
            w = cand
            break
    assert w is not None, f"no head count refuses on {sms} SMs"
    inp = I.generate(w)
    step = Step(w, workspace=False)
    step.prefill(inp)
    q, k, v = step.device_inputs(inp)
    nodes, _ = step.node_table()
    step.cache.rope_kv_write(nodes, k, v, q, check=False)
    out = torch.full((w.n_nodes, w.T, w.H, w.d), 7.0, dtype=torch.bfloat16, device="cuda")
    assert _noalloc(step, nodes, q, out, None) == sva.ERR_CAPACITY
    assert "scratch" in sva.last_error()
    torch.cuda.synchronize()
    assert bool((out == 7.0).all())                # nothing was launched
    assert step.cache.poll() == sva.OK
    # The limit is that of the wave-filling split: the plan itself does not
    # split this launch, which leaves a workspace as it was.
    ws = torch.empty(step.cache.workspace_bytes(), dtype=torch.uint8, device="cuda")
    step.cache.set_workspace(ws)
    ws.fill_(0xA5)
    step.cache.attend_nodes(nodes, q, out, None, step.scale)
    assert step.cache.poll() == sva.OK
    assert bool((ws == 0xA5).all()) and not bool((out == 7.0).all())
    step.close()


def test_plan_mirror_on_152_sms():
    """The wave-filling splits used above, on the GB300's 152 SMs: clean1 has 152
    units whole and the other 76 two ways (about 20 MB of scratch), merge4 152
    and 8 four ways."""
    w = I.WORKLOADS["clean1"]
    units = w.H * -(-w.tiles // 2)
    assert units == 228 and _plan(units, 4 * w.tiles, 152, 4 * 152) == (152, 2)
    n_split, need = _scratch(w, 152)
    assert _plan(160, 16, 152, 4 * 152) == (152, 4)
    assert n_split == 2 and need == 512 + 76 * 2 * 256 * (128 + 2) * 4   # counters + partials


_CAPTURE = """
import torch
from paper_2609_22283_gb300 import inputs as I
from paper_2609_22283_gb300 import sva
from paper_2609_22283_gb300.pipeline import Step
from tests.test_zz_no_alloc import SPLIT4, _noalloc

def ready(w):
    step, inp = Step(w, workspace=False), I.generate(w)
    step.prefill(inp)
    q, k, v = step.device_inputs(inp)
    nodes, _ = step.node_table()
    step.cache.rope_kv_write(nodes, k, v, q, check=False)
    return step, nodes, q, *step.outputs()

small, large = ready(SPLIT4), ready(I.WORKLOADS["clean1"])
torch.cuda.synchronize()
assert _noalloc(*small) == sva.OK, sva.last_error()      # the first call on the device
torch.cuda.synchronize()
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g):
    free = torch.cuda.mem_get_info()[0]
    st = _noalloc(*large)
    taken = free - torch.cuda.mem_get_info()[0]
assert st == sva.OK, sva.last_error()
assert taken == 0, f"the captured call took {taken} bytes of device memory"
g.replay()
assert large[0].cache.poll() == sva.OK
got = large[3].clone(), large[4].clone()
assert _noalloc(*large) == sva.OK
torch.cuda.synchronize()
assert torch.equal(got[0], large[3]) and torch.equal(got[1], large[4])
print("captured")
"""


def test_first_call_readies_a_capture():
    """The first call on a device, small enough to use no scratch, looks the
    scratch up all the same, so that a later call that does use it can be
    captured and takes no device memory.  In a process of its own: the look-up
    is made once per process."""
    r = subprocess.run([sys.executable, "-c", _CAPTURE], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "captured" in r.stdout, r.stderr[-2000:]

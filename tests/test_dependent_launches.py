"""Kernels of successive calls overlap (a kernel may start while the one before it runs): what that order relies on, and
calls enqueued back to back without a synchronisation in between against the same calls drained one by one."""
import os
import re

import numpy as np
import pytest
import torch

from paper_2608_07524_b200 import binding as B
from paper_2608_07524_b200 import inputs

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_07524_b200", "csrc")


def kernel_bodies():
    """(file, name, text from one kernel's head to the next's) of every kernel in the sources."""
    for fn in sorted(os.listdir(CSRC)):
        if not fn.endswith(".cu"):
            continue
        with open(os.path.join(CSRC, fn)) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        heads = [m.start() for m in re.finditer(r"__global__", text)] + [len(text)]
        for a, b in zip(heads, heads[1:]):
            yield fn, re.search(r"(\w+_kernel)\b", text[a:b]).group(1), text[a:b]


def test_tensor_memory_is_allocated_before_dependents_may_start():
    """A dependent's CTA holds its tensor memory until the grid before it has ended, and an allocation waits without limit:
    a kernel that let its dependents start first could wait for columns of a CTA that waits for it."""
    seen = 0
    for fn, name, body in kernel_bodies():
        alloc = [m.start() for m in re.finditer(r"\btmem_alloc(_pair)?\(", body)]
        if not alloc:
            continue
        seen += 1
        trigger = [m.start() for m in re.finditer(r"\bgrid_trigger\(\)", body)]
        assert len(trigger) == 1 and len(alloc) == 1, (fn, name)
        between = body[alloc[0]:trigger[0]]
        assert alloc[0] < trigger[0] and "__syncthreads();" in between, f"{fn}: {name} triggers before its allocation is complete"
    assert seen == 5, seen


def test_every_dependent_kernel_waits_for_the_ones_before_it():
    """A kernel that ended without waiting would let the next one see an unfinished predecessor of both."""
    for fn, name, body in kernel_bodies():
        n = body.count("grid_trigger();")
        if n:
            # once, at the kernel's own level, and with no way out before it
            assert n == 1 and len(re.findall(r"\n    grid_wait\(\);", body)) == 1, (fn, name)
            assert not re.search(r"\breturn;", body[:body.index("grid_wait();")]), (fn, name)


# batches that take different kernels: list with a table and the multi-tile kernels; single-tile kernels alone and beside
# the others; pairs with and without an accumulator; the short-sequence kernels
CALLS = [
    ([300, 17, 90, 256, 129], 2, 64, True), ([100] * 150, 4, 64, False), ([13, 1, 7, 32] * 40, 4, 128, False),
    ([900, 40, 300], 4, 128, False), ([200, 130, 7] * 60, 4, 72, True), ([200, 60, 128, 1] * 60, 4, 64, False),
    ([5, 9, 2], 2, 64, True), ([1500], 3, 128, True), ([64] * 300, 2, 128, True), ([700, 1, 0, 250], 4, 64, False),
]


class Call:
    def __init__(self, i, lengths, H, d, causal):
        cu = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
        self.T, self.n, self.H, self.d, self.causal, self.longest = int(cu[-1]), len(lengths), H, d, causal, max(lengths)
        self.q, self.k, self.v, self.g = (x.cuda() for x in inputs.make_qkvg(self.T, H, d, 900 + i))
        self.cu = torch.tensor(cu, device="cuda")
        self.exact_dq = self.longest <= 128 or (d > 64 and self.longest <= 256)      # no fp32 atomics

    def run(self, ws):
        o, lse = B.dcp_varlen_attn_fwd(self.q, self.k, self.v, self.cu, self.longest, self.causal, workspace=ws)
        return (o, lse) + tuple(B.dcp_varlen_attn_bwd(self.q, self.k, self.v, o, self.g, lse, self.cu, self.longest, self.causal,
                                                      workspace=ws))

    def check(self, got, ref, what):
        for name, a, b in zip(("o", "lse", "dq", "dk", "dv"), got, ref):
            if name == "dq" and not self.exact_dq:
                assert float((a.float() - b.float()).abs().max()) <= 2e-2, (what, name)      # atomics: order may differ
            else:
                assert torch.equal(a, b), (what, name)


@pytest.fixture(scope="module")
def calls():
    out = [Call(i, *c) for i, c in enumerate(CALLS)]
    need = max(B.dcp_varlen_attn_workspace(c.T, c.n, c.H, c.d)[1] for c in out)
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    refs = []
    for c in out:
        refs.append(c.run(ws))
        B.dcp_query_status(ws)                       # synchronises: nothing of one call is left when the next begins
    return out, refs, need


@pytest.mark.gpu
def test_calls_back_to_back_on_one_workspace(calls):
    cases, refs, need = calls
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    rng = np.random.default_rng(3)
    order = [int(i) for i in np.concatenate([rng.permutation(len(cases)) for _ in range(6)])]
    got = [cases[i].run(ws) for i in order]
    B.dcp_query_status(ws)
    for i, r in zip(order, got):
        cases[i].check(r, refs[i], CALLS[i])


@pytest.mark.gpu
def test_calls_back_to_back_on_two_streams(calls):
    cases, refs, need = calls
    lanes = [(torch.cuda.Stream(), torch.empty(need, dtype=torch.uint8, device="cuda")) for _ in range(2)]
    torch.cuda.synchronize()
    rng = np.random.default_rng(4)
    order = [int(i) for i in np.concatenate([rng.permutation(len(cases)) for _ in range(6)])]
    got = []
    for n, i in enumerate(order):
        stream, ws = lanes[n % 2]
        with torch.cuda.stream(stream):
            got.append(cases[i].run(ws))
    for stream, ws in lanes:
        B.dcp_query_status(ws, stream)
    for i, r in zip(order, got):
        cases[i].check(r, refs[i], CALLS[i])


@pytest.mark.gpu
def test_calls_captured_in_a_graph(calls):
    cases, refs, need = calls
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        got = [c.run(ws) for c in cases]
    for _ in range(3):
        for r in got:
            for x in r:
                x.fill_(7.0)
        graph.replay()
        torch.cuda.synchronize()
        B.dcp_query_status(ws)
        for c, r, ref in zip(cases, got, refs):
            c.check(r, ref, (c.T, c.d))

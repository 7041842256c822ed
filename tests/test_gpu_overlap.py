"""Calls that overlap on two streams choose their scales from their own "+1"
pass: max_ij U_ij, which the column budget comes from, is a word of each call.

Two branches of a captured graph run a dozen calls each side by side.  The one
problem has U of the order of k, the other U just above 1, so a budget taken
from the other call is five bits off, and C's last bits with it.
"""
import pytest

from helpers import ensure_built

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def oz():
    ensure_built()
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_06510_gb300 as oz
    oz.lib()
    return oz


def operands(m, n, k, dominant, seed):
    """Uniform entries; with `dominant` 2^-8 of that beside one 1 to a row of A
    and a column of B, all at the same k."""
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    A = torch.rand((k, m), dtype=torch.float64, device="cuda", generator=g).t() - 0.5
    B = torch.rand((n, k), dtype=torch.float64, device="cuda", generator=g).t() - 0.5
    if dominant:
        A *= 2.0 ** -8
        B *= 2.0 ** -8
        A[:, 0] = 1.0
        B[0, :] = 1.0
    return colmajor(A), colmajor(B)


def colmajor(t):
    return t.t().contiguous().t()


@pytest.mark.parametrize("entry", ["ex", "dgemm", "scale"])
@pytest.mark.parametrize("m,n,k", [(300, 270, 2000), (700, 20, 26000), (256, 256, 60)])
def test_each_call_has_its_own_column_budget(oz, entry, m, n, k):
    import torch
    calls = 12
    problems = [operands(m, n, k, dominant, 500 + dominant) for dominant in (False, True)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    if entry == "scale":
        scans = [oz.oz2_scan(A, B) for A, B in problems]
    spaces = [torch.empty(oz.oz2_workspace_size(m, n, k, 12), dtype=torch.uint8, device="cuda") for _ in problems]

    def call(i, C, stream=None):
        A, B = problems[i]
        if entry == "dgemm":
            oz.oz2_dgemm(A, B, C, stream=stream)
        elif entry == "ex":
            oz.oz2_dgemm_ex(A, B, C, workspace=spaces[i], stream=stream)
        else:
            with torch.cuda.stream(stream or torch.cuda.current_stream()):  # its outputs belong to that stream
                d, e = oz.oz2_scale(A, B, *scans[i])[3:]
                C[:, 0].copy_(d)
                C[0, 1:].copy_(e[1:])

    new = lambda: torch.zeros((n, m), dtype=torch.float64, device="cuda").t()
    want = [new() for _ in problems]
    for i in range(2):
        call(i, want[i])
        torch.cuda.synchronize()
    assert not torch.equal(want[0], want[1])
    out = [[new() for _ in range(calls)] for _ in problems]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        here = torch.cuda.current_stream()
        for s in streams:
            s.wait_stream(here)
        for c in range(calls):
            for i, s in enumerate(streams):
                call(i, out[i][c], s)
        for s in streams:
            here.wait_stream(s)
    for _ in range(8):
        for outs in out:
            for C in outs:
                C.zero_()
        graph.replay()
        torch.cuda.synchronize()
        for i in range(2):
            for c in range(calls):
                assert torch.equal(out[i][c].t().view(torch.int64), want[i].t().view(torch.int64)), (i, c)
    assert oz.oz2_check_device_status() == 0

"""A workspace that cannot be had with room for the split skinny operand of FP32
products (test hook "test_arena_limit": workspaces above it fail as the
allocation would): the calls run without it, with the same bits."""
import pytest
import torch

from paper_2209_12464_gb300 import ruqlp

pytestmark = pytest.mark.gpu

m, n, k, p, q = 3000, 2000, 64, 8, 1
d = k + p


@pytest.fixture()
def h():
    h = ruqlp.Handle(0, torch.cuda.current_stream().cuda_stream)
    yield h
    h.close()


def _inputs():
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    A = torch.randn(m, n, generator=g, device="cuda")
    return A, torch.randn(n, d, generator=g, device="cuda", dtype=torch.float64)


def _same(a, b):
    assert all(torch.equal(x, y) for x, y in zip(a[:3], b[:3]))


def test_single_calls(h):
    A, Om = _inputs()
    want = h.decompose(A, Om, k, p, q)
    Y = h.sketch(A, Om.float())
    tight = ruqlp.Handle(0, torch.cuda.current_stream().cuda_stream)
    try:
        room = ruqlp.ruqlp_workspace_bytes(m, n, d, ruqlp.F32)
        tight.set_option("test_arena_limit", room - 1)
        with pytest.raises(ruqlp.RuqlpError):
            tight.decompose(A, Om, k, p, q)
        tight.set_option("test_arena_limit", room)
        assert ruqlp.ruqlp_reserve(tight.h, m, n, d, ruqlp.F32) == ruqlp.OK
        _same(tight.decompose(A, Om, k, p, q), want)
        assert torch.equal(tight.sketch(A, Om.float()), Y)
        # the host entry: its own buffers follow the workspace
        host = m * n * 4 + n * d * 8 + (m + n + d) * d * 4 + 6 * 256
        tight.set_option("test_arena_limit", room + host)
        outs = [torch.empty(s, d) for s in (m, d, n)]
        tight.decompose_host(A.cpu(), Om.cpu(), k, p, q, outs)
        _same([t.cuda() for t in outs], want)
        tight.set_option("test_arena_limit", 0)
        _same(tight.decompose(A, Om, k, p, q), want)
    finally:
        tight.close()


def test_batch(h):
    A, Om = _inputs()
    As = [A[: 700 + 100 * i, : 600 + 50 * i].contiguous() for i in range(6)]
    Oms = [Om[: a.shape[1]].contiguous() for a in As]
    want = [tuple(t.clone() for t in r[:3]) for r in h.decompose_batch(As, Oms, [k] * 6, p, q)]
    tight = ruqlp.Handle(0, torch.cuda.current_stream().cuda_stream)
    try:
        b = tight.prepare_batch(As, Oms, [k] * 6, p, q)
        lo, hi = 1, 1 << 30  # the least workspace that the batch runs in
        while hi - lo > 1:
            mid = (lo + hi) // 2
            one = ruqlp.Handle(0, torch.cuda.current_stream().cuda_stream)
            one.set_option("test_arena_limit", mid)
            try:
                one.prepare_batch(As, Oms, [k] * 6, p, q).run()
                hi = mid
            except ruqlp.RuqlpError:
                lo = mid
            finally:
                one.close()
        tight.set_option("test_arena_limit", hi)
        for _ in range(3):  # eager, captured, replayed
            for o in b.outs:
                for t in o:
                    t.fill_(float("nan"))
            b.run()
            for o, w in zip(b.outs, want):
                _same(o, w)
    finally:
        tight.close()

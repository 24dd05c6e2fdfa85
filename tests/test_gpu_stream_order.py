"""Calls read every input in stream order, weights included: what the kernel
directly ahead of a call writes is what the call reads, also where that kernel
lets the next launch start before it ends.  The library's own rotary kernel is
such a kernel: it triggers its dependents at its start and writes the caches
afterwards.  Here the value cache it writes is the next call's weight."""
import pytest
import torch

from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def moe():
    need_gpu()
    from paper_2506_23635_gb300 import moe as m
    return m


class Writer:
    """moe_sa_qkv calls that leave n bf16 values in a value cache, in their
    last kernel (the positions in falling order, so that the first weights are
    written by its last blocks)."""

    def __init__(self, m, n):
        L = (n + 127) // 128
        assert L <= 65536
        self.m, self.n = m, n
        g = torch.Generator().manual_seed(n)
        self.a = m.sa_dims(64, 1, 1, 128, 10000.0)
        self.x = torch.randn(L, 64, generator=g).bfloat16().cuda()
        self.w = (torch.randn(3 * 128, 64, generator=g) * 0.01).bfloat16().cuda()
        self.seq = torch.zeros(L, dtype=torch.int32, device="cuda")
        self.pos = torch.arange(L - 1, -1, -1, dtype=torch.int32, device="cuda")
        self.kc = torch.empty(1, 1, L, 128, dtype=torch.bfloat16, device="cuda")
        self.vc = torch.empty_like(self.kc)
        self.ws = torch.empty(m.sa_workspace_size(self.a, L), dtype=torch.uint8, device="cuda")

    def weight(self, *shape):
        return self.vc.view(-1)[:self.n].view(*shape)

    def write(self):
        self.m.sa_qkv(self.a, self.x, self.w, self.seq, self.pos, self.kc, self.vc, ws=self.ws)


def _check(m, writer, fn):
    """fn() right behind the writer gives what it gives once the weight is there."""
    writer.write()
    torch.cuda.synchronize()
    want = [t.clone() for t in fn()]
    for _ in range(5):
        writer.vc.zero_()
        torch.cuda.synchronize()
        writer.write()
        got = fn()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, want))
    assert m.get_last_error() == 0


@pytest.mark.parametrize("T", [5, 128, 700])
def test_router_weight_written_just_ahead(T):
    m = moe()
    D, E, K = 6144, 16, 4
    wr = Writer(m, D * E)
    d = m.dims(D, 64, E, K, torch.bfloat16)
    x = torch.randn(T, D, generator=torch.Generator().manual_seed(T)).bfloat16().cuda()
    _check(m, wr, lambda: m.route(d, x, wr.weight(D, E), want_logits=True))


@pytest.mark.parametrize("T", [1, 3, 30, 200])
def test_layer_router_weight_written_just_ahead(T):
    """One token, the one-CTA and the cluster router, and the tensor cores."""
    m = moe()
    D, F, E, K = 2048, 64, 16, 4
    g = torch.Generator().manual_seed(T)
    wr = Writer(m, D * E)
    d = m.dims(D, F, E, K, torch.bfloat16)
    x = torch.randn(T, D, generator=g).bfloat16().cuda()
    w1, v1 = ((torch.randn(E, F, D, generator=g) * 0.02).bfloat16().cuda() for _ in range(2))
    w2 = (torch.randn(E, D, F, generator=g) * 0.02).bfloat16().cuda()
    ws, out = m.alloc_workspace(d, T), torch.empty(T, D, dtype=torch.bfloat16, device="cuda")
    _check(m, wr, lambda: [m.layer_forward(d, x, wr.weight(D, E), w1, v1, w2, out=out, ws=ws)])


@pytest.mark.parametrize("D,Hq,Hkv,T", [(256, 2, 1, 3), (256, 2, 1, 150), (328, 12, 4, 400),
                                        (328, 40, 8, 530), (256, 2, 1, 700)])
def test_projection_weight_written_just_ahead(D, Hq, Hkv, T):
    """The attention block's W_qkv, on each kernel that takes it: the
    weights-as-M kernel of one run of tokens and of two, the pair GEMM in equal
    shares of the (unit, k-block)s and in whole units."""
    m = moe()
    g = torch.Generator().manual_seed(T)
    wr = Writer(m, (Hq + 2 * Hkv) * 128 * D)
    a = m.sa_dims(D, Hq, Hkv, 128, 10000.0)
    x = torch.randn(T, D, generator=g).cuda()
    w_o = (torch.randn(D, Hq * 128, generator=g) * 0.02).bfloat16().cuda()
    seq = torch.zeros(T, dtype=torch.int32, device="cuda")
    pos = torch.arange(T, dtype=torch.int32, device="cuda")
    kc = torch.empty(1, Hkv, T, 128, dtype=torch.bfloat16, device="cuda")
    vc, out = torch.empty_like(kc), torch.empty_like(x)
    ws = torch.empty(m.sa_workspace_size(a, T), dtype=torch.uint8, device="cuda")
    w_qkv = wr.weight((Hq + 2 * Hkv) * 128, D)

    def block():
        m.sa_forward(a, out, w_qkv, w_o, seq, pos, kc, vc, ws=ws)
        return [out, kc, vc]

    wr.write()
    torch.cuda.synchronize()
    out.copy_(x)
    want = [t.clone() for t in block()]
    for _ in range(5):
        wr.vc.zero_()
        out.copy_(x)
        torch.cuda.synchronize()
        wr.write()
        got = block()
        torch.cuda.synchronize()
        # (the caches hold the projection itself; the block's sums over
        # positions may take their parts in another order)
        assert torch.equal(got[1], want[1]) and torch.equal(got[2], want[2])
        assert float((got[0] - want[0]).norm()) <= 1e-2 * float((want[0] - x).norm())
    assert m.get_last_error() == 0

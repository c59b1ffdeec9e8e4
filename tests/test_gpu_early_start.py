"""Kernels that start under the launch before them: a chain of the library's own calls in which each
reads what the one before wrote, with nothing between, gives the bits of the same chain with a
synchronisation after every call.  Buffers are reused from turn to turn, so that a read before the
producer's last write, or a write before the reader's last read, shows as another turn's values."""
import pytest
import torch

from paper_2604_00754_b200 import binding as sa

pytestmark = pytest.mark.gpu

CASES = [
    (1, 8, 2, 700, 128, 256, torch.bfloat16),      # less than one item per SM
    (4, 12, 12, 1024, 64, 128, torch.bfloat16),    # several
    (1, 4, 1, 17000, 64, 200, torch.bfloat16),     # the permutation's four launches
    (1, 4, 2, 600, 64, 64, torch.float32),
    (1, 4, 2, 32768 + 200, 64, 1024, torch.bfloat16),    # the SA branch over key lists
]


class Chain:
    def __init__(self, B, Hq, Hkv, n, d, w, dtype):
        g = torch.Generator(device="cuda").manual_seed(n)
        self.shape, self.w = (B, n), w
        mk = lambda h: torch.randn(B, h, n, d, generator=g, device="cuda").to(dtype)
        self.inputs = [(mk(Hq), mk(Hkv), mk(Hkv), mk(Hq)) for _ in range(2)]
        self.logits = torch.randn(2, Hq, generator=g, device="cuda")
        self.table = sa.sa_rope_table(n, d)
        self.wg = (torch.randn(Hq * d, Hq * d, generator=g, device="cuda") * (Hq * d) ** -0.5).to(dtype)
        self.q, self.k, self.v, self.dy = (torch.empty_like(t) for t in self.inputs[0])
        self.perm = torch.empty(B, n, dtype=torch.int32, device="cuda")
        self.inv = torch.empty_like(self.perm)
        self.ws = torch.empty(sa.sa_workspace_bytes(sa.SaProblem(B=B, n=n), sa.OP_MAKE_PERM),
                              dtype=torch.uint8, device="cuda")

    def turn(self, i, after=lambda: None):
        q0, k0, v0, dy0 = self.inputs[i % 2]
        turned = lambda x, out, kv: (sa.sa_rope_apply(x, q0 if kv else k0, *self.table, out=out, kv=kv), after())
        sa.sa_make_perm(7, i, *self.shape, perm=self.perm, inv=self.inv, ws=self.ws)
        after()
        turned(q0, self.q, False)
        turned(k0, self.k, True)
        turned(v0, self.v, True)
        out = sa.sa_swa_gated_forward(self.q, self.k, self.v, self.perm, self.inv, self.logits, self.w,
                                      save_for_bwd=True)
        after()
        turned(dy0, self.dy, False)
        grads = sa.sa_backward(self.q, self.k, self.v, self.perm, self.inv, self.logits, *out[1:], self.dy,
                               self.w)
        after()
        rows = grads[0].reshape(-1, self.wg.shape[0])
        gated = sa.sa_gate_projection_forward(rows, self.wg)
        after()
        back = sa.sa_gate_projection_backward(gated, rows, self.wg)
        after()
        alone = sa.sa_forward(self.q, self.k, self.v, self.perm, self.inv, self.w)
        after()
        return tuple(out) + tuple(grads) + (gated,) + tuple(back) + (alone,)


@pytest.mark.parametrize("case", CASES)
def test_chain_of_calls_with_nothing_between(case):
    chain = Chain(*case)
    got = [chain.turn(i) for i in range(6)]
    assert sa.sa_read_status() == 0
    for i, turn in enumerate(got):
        for a, b in zip(turn, chain.turn(i, torch.cuda.synchronize)):
            assert torch.equal(a, b)
    assert sa.sa_read_status() == 0


# the same launches as nodes of a graph
@pytest.mark.parametrize("case", CASES)
def test_captured_chain(case):
    chain = Chain(*case)
    chain.turn(0)                                   # kernels are loaded before the capture
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        got = [chain.turn(i) for i in range(2)]
    for _ in range(2):
        graph.replay()
        torch.cuda.synchronize()
        for i, turn in enumerate(got):
            for a, b in zip(turn, chain.turn(i, torch.cuda.synchronize)):
                assert torch.equal(a, b)
    assert sa.sa_read_status() == 0

"""Edges of the tensor-core attention kernels (128-row tiles, 64- or 128-key blocks, persistent
CTAs that run one launch into the next) and of the projection gates' split dW, bf16, against the
float64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2604_00754_b200 import binding as sa
from paper_2604_00754_b200.workloads import CAUSAL, LINEAR_WINDOW, SWA_ONE_SIDED, as_f64

pytestmark = pytest.mark.gpu

ONE = CAUSAL | SWA_ONE_SIDED

# n around a row tile; windows that end on and around 32 columns (one mask word), a 64-key and a
# 128-key block; one, two and three column tiles per row tile; every query head of a group; the
# band around the whole sequence; and more items than SMs, so that CTAs take several (3 * 8 * 8)
CASES = [
    (1, 2, 1, 127, 64, 31, ONE), (1, 2, 2, 128, 64, 33, CAUSAL), (1, 3, 1, 129, 128, 32, ONE),
    (2, 2, 1, 255, 128, 64, 0), (1, 4, 4, 256, 64, 65, CAUSAL | LINEAR_WINDOW),
    (1, 4, 2, 257, 128, 127, ONE), (1, 2, 1, 384, 64, 128, ONE), (1, 4, 1, 385, 128, 129, ONE),
    (1, 2, 1, 300, 64, 299, CAUSAL), (1, 2, 2, 300, 128, 600, ONE),
    (3, 8, 8, 900, 64, 96, ONE), (3, 16, 8, 900, 128, 200, ONE | LINEAR_WINDOW),
]


# bf16 inputs, probabilities and results with fp32 sums: 2e-2 of the largest value, as for the
# other bf16 comparisons; 1e-5 for values that cancel to zero
def _close(got, want, name):
    err = np.abs(as_f64(got) - want).max()
    assert err <= 2e-2 * np.abs(want).max() + 1e-5, (name, float(err))


@pytest.mark.parametrize("B,Hq,Hkv,n,d,w,flags", CASES)
def test_gated_pass_at_tile_edges(B, Hq, Hkv, n, d, w, flags):
    g = torch.Generator().manual_seed(n + w)
    mk = lambda h: torch.randn(B, h, n, d, generator=g).bfloat16()
    q, k, v, dy = mk(Hq), mk(Hkv), mk(Hkv), mk(Hq)
    lg = torch.randn(2, Hq, generator=g)
    perm, inv = sa.sa_make_perm(n, w, B, n)
    dev = [t.cuda() for t in (q, k, v)]
    runs = []
    for _ in range(2):
        out = sa.sa_swa_gated_forward(*dev, perm, inv, lg.cuda(), w, flags, save_for_bwd=True)
        runs.append(tuple(out) + tuple(sa.sa_backward(*dev, perm, inv, lg.cuda(), *out[1:], dy.cuda(),
                                                      w, flags)))
    assert sa.sa_read_status() == 0
    for a, b in zip(*runs):                         # no atomics: bit for bit the same
        assert torch.equal(a, b)
    args = [as_f64(t) for t in (q, k, v)] + [perm.cpu().numpy(), inv.cpu().numpy(), lg.double().numpy()]
    want = tuple(oracle.gated_forward(*args, w, flags)) + tuple(oracle.backward(*args, as_f64(dy), w, flags))
    for got, ref, name in zip(runs[0], want, ("y", "y_sa", "y_swa", "lse_sa", "lse_swa", "dq", "dk", "dv",
                                              "dgate")):
        if name.startswith("lse"):                  # a sum of bf16 products in the exponent
            assert np.abs(as_f64(got) - ref).max() <= 2e-2, name
        else:
            _close(got, ref, name)


# dW in parts of the rows: as many as rows / dm allows (64 rows are one contraction step), ragged
# rows and columns, one part; 18900 x 256 runs the 128 x 256 tiles with several items per CTA
@pytest.mark.parametrize("rows,dm", [(64, 64), (129, 64), (700, 192), (1300, 320), (4100, 128), (18900, 256)])
def test_projection_gate_backward_in_parts(rows, dm):
    g = torch.Generator().manual_seed(rows + dm)
    y, dout = (torch.randn(rows, dm, generator=g).bfloat16() for _ in range(2))
    w = (torch.randn(dm, dm, generator=g) * dm ** -0.5).bfloat16()
    runs = [sa.sa_gate_projection_backward(dout.cuda(), y.cuda(), w.cuda()) for _ in range(2)]
    assert sa.sa_read_status() == 0
    want = oracle.gate_projection_backward(dout.double().numpy(), y.double().numpy(), w.double().numpy())
    for got, again, ref, name in zip(*runs, want, ("dy", "dw")):
        assert torch.equal(got, again)
        _close(got, ref, name)


# pieces of whole sequences, of one head range per sequence range, and of several; odd lengths, so
# that a range's index lists start off 16 bytes
@pytest.mark.parametrize("B,Hq,Hkv,n", [(5, 8, 2, 1001), (3, 16, 4, 1003), (2, 16, 8, 1501), (9, 2, 2, 2002)])
def test_host_pieces_of_a_batch(B, Hq, Hkv, n):
    from paper_2604_00754_b200.host import HostForward
    g = torch.Generator().manual_seed(n)
    q, k, v = (torch.randn(B, h, n, 64, generator=g).bfloat16().pin_memory() for h in (Hq, Hkv, Hkv))
    lg = torch.randn(2, Hq, generator=g).pin_memory()
    y = torch.empty_like(q).pin_memory()
    HostForward(B, Hq, Hkv, n, 64, 96).forward(q, k, v, lg, y, seed=7, layer=1)
    torch.cuda.synchronize()
    perm, inv = sa.sa_make_perm(7, 1, B, n)
    want = sa.sa_swa_gated_forward(q.cuda(), k.cuda(), v.cuda(), perm, inv, lg.cuda(), 96, ONE)
    want = want[0] if isinstance(want, (tuple, list)) else want
    assert torch.equal(y, want.cpu())
    assert sa.sa_read_status() == 0


# A sequence's result does not depend on what else is in the call: alone (at most one item per SM) and
# in a batch (several), or in a piece of the host pipeline, it has the same bits.
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("w", [128, 129, 256, 320])
def test_bits_of_a_sequence_alone_and_in_a_batch(w, d):
    g = torch.Generator().manual_seed(w)
    q, k, v = (torch.randn(8, h, 600, d, generator=g).bfloat16().cuda() for h in (16, 8, 8))
    lg = torch.randn(2, 16, generator=g).cuda()
    perm, inv = sa.sa_make_perm(3, 1, 8, 600)
    whole = sa.sa_swa_gated_forward(q, k, v, perm, inv, lg, w, save_for_bwd=True)
    part = [t[2:3].contiguous() for t in (q, k, v, perm, inv)]
    for a, b in zip(whole, sa.sa_swa_gated_forward(*part, lg, w, save_for_bwd=True)):
        assert torch.equal(a[2:3], b)
    assert sa.sa_read_status() == 0


@pytest.mark.parametrize("w", [129, 256, 320])
def test_host_pieces_have_the_bits_of_the_whole(w):
    from paper_2604_00754_b200.host import HostForward
    g = torch.Generator().manual_seed(w)
    q, k, v = (torch.randn(1, h, 2048, 128, generator=g).bfloat16().pin_memory() for h in (32, 8, 8))
    lg = torch.randn(2, 32, generator=g).pin_memory()
    y = torch.empty_like(q).pin_memory()
    HostForward(1, 32, 8, 2048, 128, w).forward(q, k, v, lg, y, seed=7, layer=1)
    torch.cuda.synchronize()
    perm, inv = sa.sa_make_perm(7, 1, 1, 2048)
    want = sa.sa_swa_gated_forward(q.cuda(), k.cuda(), v.cuda(), perm, inv, lg.cuda(), w, ONE)
    assert torch.equal(y, want.cpu())
    assert sa.sa_read_status() == 0


# the forward's choice of tiles at its lines.  One path: 74 wide tiles (half of 148), 73 x 128 rows and
# one more at dm = 256.  Two paths: 296 wide tiles at dm = 256, and sizes below them at dm = 1024
@pytest.mark.parametrize("rows,dm,dual", [(9344, 256, False), (9345, 256, False), (37889, 256, True),
                                          (2304, 1024, True), (2305, 1024, True)])
def test_projection_gate_forward_tile_choice(rows, dm, dual):
    g = torch.Generator().manual_seed(rows)
    ya, yb = (torch.randn(rows, dm, generator=g).bfloat16() for _ in range(2))
    wa, wb = ((torch.randn(dm, dm, generator=g) * dm ** -0.5).bfloat16() for _ in range(2))
    args = (ya, wa, yb, wb) if dual else (ya, wa)
    out = sa.sa_gate_projection_forward(*(t.cuda() for t in args))
    assert sa.sa_read_status() == 0
    _close(out, oracle.gate_projection(*(t.double().numpy() for t in args)), "out")


# Two paths below two wide tiles per SM: one launch, both products added in fp32 and rounded once.
# Half a unit in the last place of bf16 for the rounding, and for each path its value times 2^-11: the
# logistic is half a hardware tanh, whose relative error is 2^-11, and the rest is for the fp32 sums.
@pytest.mark.parametrize("rows,dm", [(2305, 1024), (1200, 2048), (640, 4096)])
def test_two_gate_paths_are_rounded_once(rows, dm):
    g = torch.Generator().manual_seed(rows)
    ya, yb = (torch.randn(rows, dm, generator=g).bfloat16() for _ in range(2))
    wa, wb = ((torch.randn(dm, dm, generator=g) * dm ** -0.5).bfloat16() for _ in range(2))
    out = sa.sa_gate_projection_forward(ya.cuda(), wa.cuda(), yb.cuda(), wb.cuda())
    assert sa.sa_read_status() == 0
    want = oracle.gate_projection(*(t.double().numpy() for t in (ya, wa, yb, wb)))
    half_ulp = np.exp2(np.floor(np.log2(np.abs(want) + 1e-30)) - 8)
    bound = half_ulp + 2.0 ** -11 * (as_f64(ya.abs()) + as_f64(yb.abs()))
    assert (np.abs(as_f64(out) - want) <= bound).all()

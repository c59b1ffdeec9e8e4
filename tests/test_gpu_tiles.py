"""Edges of the tiled CUDA-core kernels (32 rows x 32 columns, fp32) and of the one-launch
permutation sort, against the float64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2604_00754_b200 import binding as sa
from paper_2604_00754_b200.workloads import CAUSAL, LINEAR_WINDOW, SWA_ONE_SIDED, as_f64

pytestmark = pytest.mark.gpu


# n around a row tile, the band around the sequence (the window of a tile wraps onto itself before
# the window of a row does), every column-group count of d, split and unsplit gradients
@pytest.mark.parametrize("B,Hq,Hkv,n,d,w,flags", [
    (1, 2, 1, 31, 8, 5, CAUSAL | SWA_ONE_SIDED),
    (2, 2, 1, 32, 64, 31, CAUSAL | SWA_ONE_SIDED),
    (1, 3, 1, 33, 72, 34, CAUSAL | SWA_ONE_SIDED),
    (1, 2, 2, 97, 128, 70, 0),
    (1, 4, 2, 129, 136, 128, CAUSAL | LINEAR_WINDOW),
    (1, 2, 1, 65, 256, 64, CAUSAL | SWA_ONE_SIDED),
    (8, 8, 4, 1185, 16, 3, CAUSAL | SWA_ONE_SIDED),     # 32 * 38 key tiles: not split
    (1, 8, 1, 9473, 8, 9, CAUSAL | SWA_ONE_SIDED),      # 297: a group's heads in four parts
    (1, 6, 1, 12641, 8, 7, 0),                          # 396: in three
])
def test_fp32_tiles(B, Hq, Hkv, n, d, w, flags):
    g = torch.Generator().manual_seed(n + d)
    mk = lambda h: torch.randn(B, h, n, d, generator=g)
    q, k, v, dy = mk(Hq), mk(Hkv), mk(Hkv), mk(Hq)
    lg = torch.randn(2, Hq, generator=g)
    perm, inv = sa.sa_make_perm(n, 3, B, n)
    dev = [t.cuda() for t in (q, k, v)]
    y, y_sa, y_swa, lse_sa, lse_swa = sa.sa_swa_gated_forward(*dev, perm, inv, lg.cuda(), w, flags,
                                                              save_for_bwd=True)
    grads = sa.sa_backward(*dev, perm, inv, lg.cuda(), y_sa, y_swa, lse_sa, lse_swa, dy.cuda(), w,
                           flags)
    args = [as_f64(t) for t in (q, k, v)] + [perm.cpu().numpy(), inv.cpu().numpy(),
                                             lg.double().numpy()]
    ref = oracle.gated_forward(*args, w, flags)
    for got, want in zip((y, y_sa, y_swa, lse_sa, lse_swa), ref):
        assert np.abs(as_f64(got) - want).max() <= 1e-4
    # gradients are sums of up to band * G terms of size O(1): the fp32 bound scaled by their size
    for got, want in zip(grads, oracle.backward(*args, as_f64(dy), w, flags)):
        assert np.abs(as_f64(got) - want).max() <= 1e-4 * max(1.0, np.abs(want).max())
    assert sa.sa_read_status() == 0


# More (branch, head) pairs than a grid's second dimension has: split (two parts per group, 84000) and
# not (80000 per branch)
@pytest.mark.parametrize("Hq,Hkv,n", [(40000, 1000, 32), (40000, 40000, 8)])
def test_fp32_backward_of_many_heads(Hq, Hkv, n):
    g = torch.Generator().manual_seed(n)
    mk = lambda h: torch.randn(1, h, n, 8, generator=g)
    q, k, v, dy = mk(Hq), mk(Hkv), mk(Hkv), mk(Hq)
    lg, w, flags = torch.randn(2, Hq, generator=g), 5, CAUSAL | SWA_ONE_SIDED
    perm, inv = sa.sa_make_perm(n, 3, 1, n)
    dev = [t.cuda() for t in (q, k, v)]
    out = sa.sa_swa_gated_forward(*dev, perm, inv, lg.cuda(), w, flags, save_for_bwd=True)
    grads = sa.sa_backward(*dev, perm, inv, lg.cuda(), *out[1:], dy.cuda(), w, flags)
    assert sa.sa_read_status() == 0
    args = [as_f64(t) for t in (q, k, v)] + [perm.cpu().numpy(), inv.cpu().numpy(), lg.double().numpy()]
    for got, want in zip(grads, oracle.backward(*args, as_f64(dy), w, flags)):
        assert np.abs(as_f64(got) - want).max() <= 1e-4 * max(1.0, np.abs(want).max())


# An infinity or a NaN reaches the rows and columns that its token meets and no others, although the
# tiles hold pairs that do not see each other.  Finite where the oracle is, to the tolerances above
# (bf16: 2e-2 of the largest finite value); the rest is not finite.
@pytest.mark.parametrize("B,Hq,Hkv,n,d,dtype,flags", [
    (1, 2, 1, 300, 64, torch.float32, CAUSAL | SWA_ONE_SIDED),
    (1, 2, 2, 301, 128, torch.float32, 0),
    (8, 8, 4, 1185, 16, torch.float32, CAUSAL | LINEAR_WINDOW),     # gradients not split
    (1, 4, 2, 300, 72, torch.bfloat16, CAUSAL | SWA_ONE_SIDED),
])
def test_not_finite_values_stay_with_the_pairs_that_see_them(B, Hq, Hkv, n, d, dtype, flags):
    g = torch.Generator().manual_seed(n)
    mk = lambda h: torch.randn(B, h, n, d, generator=g).to(dtype)
    q, k, v, dy = mk(Hq), mk(Hkv), mk(Hkv), mk(Hq)
    v[:, :, 150, d // 2] = float("inf")
    k[:, :, 40] = float("nan")
    q[:, :, 250, 0] = float("nan")
    dy[:, :, 200, d - 1] = -float("inf")
    lg, w = torch.randn(2, Hq, generator=g), 9
    perm, inv = sa.sa_make_perm(n, 1, B, n)
    dev = [t.cuda() for t in (q, k, v)]
    out = sa.sa_swa_gated_forward(*dev, perm, inv, lg.cuda(), w, flags, save_for_bwd=True)
    grads = sa.sa_backward(*dev, perm, inv, lg.cuda(), *out[1:], dy.cuda(), w, flags)
    assert sa.sa_read_status() == 0
    args = [as_f64(t) for t in (q, k, v)] + [perm.cpu().numpy(), inv.cpu().numpy(), lg.double().numpy()]
    want = tuple(oracle.gated_forward(*args, w, flags))[:3] + \
        tuple(oracle.backward(*args, as_f64(dy), w, flags))[:3]
    for got, ref, name in zip(out[:3] + tuple(grads[:3]), want, ("y", "y_sa", "y_swa", "dq", "dk", "dv")):
        got, finite = as_f64(got), np.isfinite(ref)
        assert finite.mean() > 0.4 and not finite.all(), name
        assert np.array_equal(np.isfinite(got), finite), name
        err, top = np.abs(got[finite] - ref[finite]).max(), np.abs(ref[finite]).max()
        assert err <= (1e-4 * max(1.0, top) if dtype == torch.float32 else 2e-2 * top), name


# one CTA up to 1024 tokens, clusters of 2, 4 and 8 up to 16384, global memory beyond
@pytest.mark.parametrize("B,n", [(2, 33), (1, 1024), (2, 1025), (1, 2049), (3, 4097), (2, 8191),
                                 (1, 16384), (1, 16385)])
def test_make_perm_cluster_sizes(B, n):
    perm, inv = sa.sa_make_perm(0x123456789ABCDEF0 + n, 5, B, n)
    operm, oinv = oracle.make_perm(0x123456789ABCDEF0 + n, 5, B, n)
    assert np.array_equal(perm.cpu().numpy(), operm)
    assert np.array_equal(inv.cpu().numpy(), oinv)

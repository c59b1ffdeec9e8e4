"""The causal SA branch over token-ordered key lists (wide windows, long sequences, an even number of
query heads per KV head): rows against the float64 oracle, and against the same kernels without
lists."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2604_00754_b200 import binding as sa
from paper_2604_00754_b200.workloads import CAUSAL, LINEAR_WINDOW, SWA_ONE_SIDED, as_f64

# groups of 256 and of 512 slots (w from 1281 on); last groups of one slot, of less than a tile, of an
# odd number of tiles; both head dimensions; windows that wrap and windows that end with the sequence
CASES = [
    (1, 2, 1, 32768, 128, 1024, CAUSAL), (1, 4, 2, 32769, 64, 1280, CAUSAL),
    (2, 2, 1, 32768 + 200, 64, 1025, CAUSAL | LINEAR_WINDOW), (1, 2, 1, 32768 + 300, 128, 1281, CAUSAL),
    (1, 4, 1, 33000, 128, 2048, CAUSAL | LINEAR_WINDOW), (1, 2, 1, 32768 + 385, 64, 7000, CAUSAL),
]


def problem(Hq, Hkv, n, d, w, flags, B=1, dtype=sa.BF16):
    p = sa.SaProblem(B=B, Hq=Hq, Hkv=Hkv, n=n, d=d, w=w, dtype=dtype, flags=flags)
    sa.load_library().sa_problem_set_contiguous(ctypes.byref(p))
    return p


def test_which_problems_use_lists():
    size = lambda *a, **k: sa.sa_workspace_bytes(problem(*a, **k), sa.OP_KEY_LISTS)
    assert size(2, 1, 32768, 128, 1024, CAUSAL) > 32768 * 4
    assert size(4, 2, 32768, 64, 1024, CAUSAL, B=2) == 2 * size(4, 2, 32768, 64, 1024, CAUSAL)
    assert size(2, 1, 32768, 128, 1024, 0) == 0                        # nothing is hidden by token
    assert size(2, 2, 32768, 128, 1024, CAUSAL) == 0                   # no two heads share a stream
    assert size(2, 1, 32768, 128, 1024, CAUSAL, dtype=sa.F32) == 0
    assert size(2, 1, 32768, 128, 32768, CAUSAL) == 0                  # a group's window over everything
    assert size(2, 1, 32767, 128, 1024, CAUSAL) == size(2, 1, 32768, 128, 1023, CAUSAL) == 0
    with pytest.raises(sa.SaError):
        sa.sa_workspace_bytes(problem(3, 2, 32768, 128, 1024, CAUSAL), sa.OP_KEY_LISTS)


@pytest.mark.gpu
@pytest.mark.parametrize("B,Hq,Hkv,n,d,w,flags", CASES)
def test_rows_against_the_oracle(B, Hq, Hkv, n, d, w, flags):
    g = torch.Generator().manual_seed(n + w)
    q, k, v = (torch.randn(B, h, n, d, generator=g).bfloat16() for h in (Hq, Hkv, Hkv))
    dev = [t.cuda() for t in (q, k, v)]
    perm, inv = sa.sa_make_perm(n, w, B, n)
    y, lse = sa.sa_forward(*dev, perm, inv, w, flags, want_lse=True)
    again = sa.sa_forward(*dev, perm, inv, w, flags)
    assert torch.equal(y, again)
    # the same call without scratch: every block of the window in slot order
    p = sa.make_problem(dev[0], dev[1], w, flags)
    plain, plse = torch.empty_like(y), torch.empty_like(lse)
    at = lambda t: ctypes.c_void_p(t.data_ptr())
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert sa.load_library().sa_forward(ctypes.byref(p), *map(at, dev), at(perm), at(inv), at(plain), at(plse),
                                        None, 0, st) == 0
    assert sa.sa_read_status() == 0
    assert not torch.equal(y, plain)
    # two roundings of P and one of y on either side, each 2^-9 of a row's largest weight or value at most
    assert (y.float() - plain.float()).norm() <= 1e-2 * plain.float().norm()
    assert (lse - plse).abs().max() <= 1e-4            # fp32 sums of the same terms in another order
    permc, invc = perm.cpu().numpy(), inv.cpu().numpy()
    rng = np.random.default_rng(0)
    # random rows, the first and last tokens, and the tokens of the first and last slots (the last group)
    tokens = np.concatenate([[0, 1, n - 1], permc[-1, :2], permc[-1, -140:]])
    rows = np.unique(np.concatenate([rng.integers(0, B * Hq * n, 1500), (B * Hq - 1) * n + tokens]))
    ry, rl = oracle.forward_rows(0, *(as_f64(t) for t in (q, k, v)), permc, invc, w, flags, rows)
    sel = torch.from_numpy(rows).cuda()
    assert np.abs(as_f64(y.reshape(-1, d)[sel]) - ry).max() <= 2e-2 * np.abs(ry).max()
    assert np.abs(as_f64(lse.reshape(-1)[sel]) - rl).max() <= 2e-2


# The host pipeline has the bits of the call on the whole problem: lists that do not fit within the scratch
# it needs otherwise; ranges of sequences, whose lists are made anew from a permutation off 16 bytes; pieces
# that cut a group to one head, whose items are two tiles of that head (a last group of one and of three tiles)
@pytest.mark.gpu
@pytest.mark.parametrize("B,Hq,Hkv,n,w,kind", [
    (1, 2, 1, 32768, 2048, "outside"), (3, 2, 1, 33001, 2000, "outside"), (2, 4, 2, 33001, 1024, "ranges"),
    (1, 4, 2, 38001, 1024, "cut"), (1, 4, 2, 38001, 2000, "cut"), (1, 4, 2, 38201, 2000, "cut"),
])
def test_bits_of_the_host_pipeline(B, Hq, Hkv, n, w, kind):
    from paper_2604_00754_b200.host import HostForward
    flags = CAUSAL | SWA_ONE_SIDED
    g = torch.Generator().manual_seed(n + w)
    q, k, v = (torch.randn(B, h, n, 64, generator=g).bfloat16().pin_memory() for h in (Hq, Hkv, Hkv))
    lg = torch.randn(2, Hq, generator=g).pin_memory()
    hf = HostForward(B, Hq, Hkv, n, 64, w, flags)
    if kind == "outside":
        assert hf.ws.numel() > sa.host_forward_ws_bytes(B, Hq, Hkv, n, 64)
    if B > 1:
        assert len({piece[5:] for piece in hf.pieces}) == B
    if kind == "cut":
        assert any((piece[3] - piece[2]) % 2 for piece in hf.pieces)
    y = torch.empty_like(q).pin_memory()
    for layer in (1, 2):
        hf.forward(q, k, v, lg, y, seed=7, layer=layer)
        torch.cuda.synchronize()
        perm, inv = sa.sa_make_perm(7, layer, B, n)
        assert torch.equal(y, sa.sa_swa_gated_forward(q.cuda(), k.cuda(), v.cuda(), perm, inv, lg.cuda(), w,
                                                      flags).cpu())
    assert sa.sa_read_status() == 0


# a part of the heads, the rotated call and the host pipeline take the same route and give the same bits
@pytest.mark.gpu
@pytest.mark.parametrize("w", [1024, 2000])
def test_bits_of_a_part_and_of_the_host_pipeline(w):
    from paper_2604_00754_b200.host import HostForward
    n, d, flags = 33100, 64, CAUSAL | SWA_ONE_SIDED
    g = torch.Generator().manual_seed(w)
    q, k, v = (torch.randn(1, h, n, d, generator=g).bfloat16().pin_memory() for h in (4, 2, 2))
    lg = torch.randn(2, 4, generator=g).pin_memory()
    dev = [t.cuda() for t in (q, k, v)]
    perm, inv = sa.sa_make_perm(7, 1, 1, n)
    whole = sa.sa_swa_gated_forward(*dev, perm, inv, lg.cuda(), w, flags, save_for_bwd=True)
    part = sa.sa_swa_gated_forward(dev[0][:, 2:], dev[1][:, 1:], dev[2][:, 1:], perm, inv,
                                   lg[:, 2:].contiguous().cuda(), w, flags, save_for_bwd=True,
                                   out={x: torch.empty_like(dev[0])[:, 2:] for x in ("y", "y_sa", "y_swa")})
    for a, b in zip(whole, part):
        assert torch.equal(a[:, 2:], b)
    cs, sn = sa.sa_rope_table(n, d, 1e6)
    turned = sa.sa_rope_apply(dev[0], dev[1], cs, sn), sa.sa_rope_apply(dev[1], dev[0], cs, sn, kv=True)
    assert torch.equal(sa.sa_forward_rope(*dev, perm, inv, cs, sn, w, CAUSAL),
                       sa.sa_forward(*turned, dev[2], perm, inv, w, CAUSAL))
    y = torch.empty_like(q).pin_memory()
    HostForward(1, 4, 2, n, d, w, flags, q_parts=2).forward(q, k, v, lg, y, seed=7, layer=1)
    torch.cuda.synchronize()
    want = sa.sa_swa_gated_forward(*dev, perm, inv, lg.cuda(), w, flags)
    assert torch.equal(y, want.cpu())
    assert sa.sa_read_status() == 0


# The attention launch looks at the status word for itself, after the launch that makes the lists, and the
# word may have been read and cleared in between: the lists are written whatever the word says, with tokens
# that exist whatever the permutation holds.
@pytest.mark.gpu
def test_lists_are_written_whatever_the_status_word_says():
    n, d, w, flags = 33000, 64, 1024, CAUSAL | 16                     # SA_VALIDATE_PERM
    g = torch.Generator(device="cuda").manual_seed(n)
    q, k, v = (torch.randn(1, h, n, d, generator=g, device="cuda").bfloat16() for h in (2, 1, 1))
    perm, inv = sa.sa_make_perm(n, w, 1, n)
    bad = perm.clone()
    bad[0, :4] = torch.tensor([n, -1, 2 ** 31 - 1, -2 ** 31])
    bad[0, 500:700] = bad[0, 700]
    p = sa.make_problem(q, k, w, flags)
    size = sa.sa_workspace_bytes(p, sa.OP_KEY_LISTS)
    at = lambda t: ctypes.c_void_p(t.data_ptr())

    def lists(sigma):
        ws, y = torch.zeros(size, dtype=torch.uint8, device="cuda"), torch.zeros_like(q)
        st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        assert sa.load_library().sa_forward_lists(ctypes.byref(p), at(q), at(k), at(v), at(sigma), at(inv), at(y),
                                                  None, at(ws), size, st) == 0
        return ws, y

    want, y = lists(perm)
    assert sa.sa_read_status() == 0 and y.any()
    rejected, y = lists(bad)
    assert not y.any()                                   # the attention launch left
    again, y = lists(perm)                               # the word is set still
    assert not y.any() and torch.equal(again, want)
    assert sa.sa_read_status() == 5                      # SA_ERR_BAD_PERM
    tiles, blocks = (n + 127) // 128, (256 + 2 * ((w + 1) // 2 - 1) + 127) // 128
    groups = (n + 255) // 256
    up = lambda x: (x + 255) // 256 * 256
    words = rejected.view(torch.int32)
    k_end = up(tiles * 512) + up(groups * blocks * 512)
    assert 0 <= words[:k_end // 4].min() and words[:k_end // 4].max() < n
    met = words[k_end // 4:k_end // 4 + tiles]
    assert 1 <= met.min() and met.max() <= blocks


def structured(kind, n):
    i = torch.arange(n, dtype=torch.int64, device="cuda")
    if kind == "identity":
        perm = i
    elif kind == "reversed":
        perm = n - 1 - i
    elif kind == "blocks":                              # shuffled blocks of 250 tokens and a ragged one
        g = torch.Generator(device="cuda").manual_seed(n)
        first = torch.randperm((n + 249) // 250, generator=g, device="cuda")
        perm = (first[:, None] * 250 + torch.arange(250, device="cuda")).reshape(-1)
        perm = perm[perm < n]
    else:                                               # strides: neighbours are 64 slots apart
        perm = torch.cat([i[s::64] for s in range(64)])
    inv = torch.empty_like(perm)
    inv[perm] = i
    return perm.int()[None].contiguous(), inv.int()[None].contiguous()


# permutations that keep neighbours together, 64 tokens and more to a bucket of the launch that makes the lists
@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["identity", "reversed", "blocks", "strides"])
@pytest.mark.parametrize("n,w,flags", [(65613, 1024, CAUSAL), (65613, 1500, CAUSAL | LINEAR_WINDOW),
                                       (70001, 7000, CAUSAL)])
def test_structured_permutations(kind, n, w, flags):
    g = torch.Generator().manual_seed(n)
    q, k, v = (torch.randn(1, h, n, 64, generator=g).bfloat16() for h in (2, 1, 1))
    dev = [t.cuda() for t in (q, k, v)]
    perm, inv = structured(kind, n)
    y, lse = sa.sa_forward(*dev, perm, inv, w, flags, want_lse=True)
    assert sa.sa_read_status() == 0
    rows = np.unique(np.concatenate([np.random.default_rng(0).integers(0, 2 * n, 600), np.arange(n - 140, n),
                                     perm[0, -80:].cpu().numpy()]))
    ry, rl = oracle.forward_rows(0, *(as_f64(t) for t in (q, k, v)), perm.cpu().numpy(), inv.cpu().numpy(), w,
                                 flags, rows)
    sel = torch.from_numpy(rows).cuda()
    assert np.abs(as_f64(y.reshape(-1, 64)[sel]) - ry).max() <= 2e-2 * np.abs(ry).max()
    assert np.abs(as_f64(lse.reshape(-1)[sel]) - rl).max() <= 2e-2


# ... and they take about the time of a random one: 1.6 times as long, and 4.3 times at n = 2^20, where the
# keys of a bucket were counted through for each of them
@pytest.mark.gpu
def test_structured_permutations_are_not_slow():
    n, w = 1 << 18, 2048
    g = torch.Generator(device="cuda").manual_seed(n)
    q, k, v = (torch.randn(1, h, n, 64, generator=g, device="cuda").bfloat16() for h in (2, 1, 1))
    times = {}
    for kind in ("random", "identity", "blocks"):
        perm, inv = sa.sa_make_perm(1, 0, 1, n) if kind == "random" else structured(kind, n)
        runs = []
        for _ in range(6):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(4):
                sa.sa_forward(q, k, v, perm, inv, w, CAUSAL)
            b.record()
            torch.cuda.synchronize()
            runs.append(a.elapsed_time(b))
        times[kind] = min(runs)
    assert sa.sa_read_status() == 0
    assert max(times["identity"], times["blocks"]) <= 1.3 * times["random"], times


# Without memory for the lists the calls work as they did without them, and say so.
@pytest.mark.gpu
def test_calls_go_without_lists_where_memory_is_short():
    from paper_2604_00754_b200.host import HostForward
    n, w, flags = 65536, 2048, CAUSAL                   # 22 MB of lists: never within another block
    g = torch.Generator(device="cuda").manual_seed(n)
    q, k, v = (torch.randn(1, h, n, 64, generator=g, device="cuda").bfloat16() for h in (2, 1, 1))
    perm, inv = sa.sa_make_perm(n, w, 1, n)
    cs, sn = sa.sa_rope_table(n, 64)
    lg = torch.zeros(2, 2, device="cuda")
    p = sa.make_problem(q, k, w, flags)
    at = lambda t: ctypes.c_void_p(t.data_ptr())
    want, y, y2, out = (torch.empty_like(q) for _ in range(4))
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert sa.load_library().sa_forward(ctypes.byref(p), at(q), at(k), at(v), at(perm), at(inv), at(want), None,
                                        None, 0, st) == 0
    copies = sa.sa_workspace_bytes(p, sa.OP_FORWARD_ROPE) - sa.sa_workspace_bytes(p, sa.OP_KEY_LISTS)
    least = sa.host_forward_ws_bytes(1, 2, 1, n, 64)
    total = torch.cuda.get_device_properties(0).total_memory
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    short = lambda spare: torch.cuda.set_per_process_memory_fraction(
        (torch.cuda.memory_reserved() + spare) / total)
    try:
        short(0)
        with pytest.warns(RuntimeWarning, match="key lists"):
            sa.sa_forward(q, k, v, perm, inv, w, flags, y=y)
        with pytest.warns(RuntimeWarning, match="key lists"):
            sa.sa_swa_gated_forward(q, k, v, perm, inv, lg, w, flags | SWA_ONE_SIDED, out={"y": out, "y_sa": y2})
        torch.cuda.empty_cache()
        short(copies + 2 * q.numel() + (4 << 20))       # ... and y
        with pytest.warns(RuntimeWarning, match="key lists"):
            sa.sa_forward_rope(q, k, v, perm, inv, cs, sn, w, flags)
        torch.cuda.empty_cache()
        short(least + (4 << 20))
        with pytest.warns(RuntimeWarning, match="key lists"):
            assert HostForward(1, 2, 1, n, 64, w, flags).ws.numel() == least
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert torch.equal(y, want) and torch.equal(y2, want)
    assert not torch.equal(sa.sa_forward(q, k, v, perm, inv, w, flags), y)
    assert sa.sa_read_status() == 0


def _lists_call(q, k, v, perm, inv, w, flags, ws, size):
    """The C call with the given scratch (None: the plain one's route)."""
    p, y = sa.make_problem(q, k, w, flags), torch.empty_like(q)
    at = lambda t: ctypes.c_void_p(t.data_ptr())
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert sa.load_library().sa_forward_lists(ctypes.byref(p), at(q), at(k), at(v), at(perm), at(inv), at(y), None,
                                              ws, size, st) == 0
    return y


# token-major tensors, checked permutations and a batch take the lists with the same bits; scratch that is too
# small, or off 16 bytes, is left alone and the call goes without
@pytest.mark.gpu
def test_layouts_checks_and_scratch():
    n, w = 33000, 1300
    g = torch.Generator(device="cuda").manual_seed(n)
    q, k, v = (torch.randn(2, h, n, 64, generator=g, device="cuda").bfloat16() for h in (4, 2, 2))
    perm, inv = sa.sa_make_perm(n, w, 2, n)
    y = sa.sa_forward(q, k, v, perm, inv, w, CAUSAL)
    major = [t.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3) for t in (q, k, v)]
    assert torch.equal(sa.sa_forward(*major, perm, inv, w, CAUSAL), y)
    assert torch.equal(sa.sa_forward(q, k, v, perm, inv, w, CAUSAL | 16), y)      # SA_VALIDATE_PERM
    one = [t[1:2].contiguous() for t in (q, k, v, perm, inv)]
    assert torch.equal(sa.sa_forward(*one, w, CAUSAL), y[1:2])
    size = sa.sa_workspace_bytes(sa.make_problem(q, k, w, CAUSAL), sa.OP_KEY_LISTS)
    ws = torch.zeros(size + 16, dtype=torch.uint8, device="cuda")
    args = (q, k, v, perm, inv, w, CAUSAL)
    plain = _lists_call(*args, None, 0)
    assert not torch.equal(plain, y)
    assert torch.equal(_lists_call(*args, ctypes.c_void_p(ws.data_ptr()), size - 1), plain)
    assert torch.equal(_lists_call(*args, ctypes.c_void_p(ws.data_ptr() + 8), size), plain)
    assert not ws.any()
    assert torch.equal(_lists_call(*args, ctypes.c_void_p(ws.data_ptr() + 16), size), y)
    assert sa.sa_read_status() == 0


# An infinity or a NaN in V: the rows that see it have it, and no row does outside the groups of 256 slots whose
# window holds it (hidden pairs within a group's blocks weigh 0, and 0 times it is a NaN).
@pytest.mark.gpu
@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_reach_of_what_is_not_finite(value):
    n, w = 33000, 1024
    g = torch.Generator(device="cuda").manual_seed(n)
    q, k, v = (torch.randn(1, h, n, 64, generator=g, device="cuda").bfloat16() for h in (2, 1, 1))
    perm, inv = sa.sa_make_perm(n, w, 1, n)
    clean = sa.sa_forward(q, k, v, perm, inv, w, CAUSAL)
    token = n // 2
    v[0, 0, token] = value
    y = sa.sa_forward(q, k, v, perm, inv, w, CAUSAL)
    assert sa.sa_read_status() == 0
    slot, h = int(inv[0, token]), (w + 1) // 2 - 1
    slots = torch.arange(n, device="cuda")
    away = lambda a, b: torch.minimum((a - b).abs(), n - (a - b).abs())
    tokens = perm[0].long()
    sees = (away(slots, slot) <= h) & (tokens >= token)
    assert sees.sum() > w // 8
    assert not torch.isfinite(y[0][:, tokens[sees]]).any()
    first = slots // 256 * 256
    last = torch.minimum(first + 255, torch.tensor(n - 1, device="cuda"))
    held = (away(first, slot) <= h) | (away(last, slot) <= h) | ((first <= slot) & (slot <= last))
    rest = tokens[~held]
    assert rest.numel() > n // 2 and torch.equal(y[0][:, rest], clean[0][:, rest])


# two query heads: rotated Q and K are below the size from which the pass is taken without lists
@pytest.mark.gpu
def test_small_rotated_call_takes_the_pass_and_lists():
    n, d, w = 32768, 64, 1024
    g = torch.Generator(device="cuda").manual_seed(n)
    q, k, v = (torch.randn(1, h, n, d, generator=g, device="cuda").bfloat16() for h in (2, 1, 1))
    assert q.numel() < 8 << 20
    perm, inv = sa.sa_make_perm(n, w, 1, n)
    cs, sn = sa.sa_rope_table(n, d, 1e6)
    turned = sa.sa_rope_apply(q, k, cs, sn), sa.sa_rope_apply(k, q, cs, sn, kv=True)
    launches = sa.launch_count()
    y = sa.sa_forward_rope(q, k, v, perm, inv, cs, sn, w, CAUSAL)
    assert sa.launch_count() - launches == 3
    assert torch.equal(y, sa.sa_forward(*turned, v, perm, inv, w, CAUSAL))
    assert sa.sa_read_status() == 0

"""Host-to-host forward: the head grouping (CPU) and, on a GPU, that the pipelined path gives
the bits of the single device-resident call."""
import pytest
import torch

from paper_2604_00754_b200 import binding as sab
from paper_2604_00754_b200 import host


def test_head_groups_cover_every_head_once():
    for Hq, Hkv, ng in [(32, 8, 8), (32, 8, 3), (12, 12, 5), (4, 1, 8), (16, 4, 1)]:
        groups = sab.host_forward_plan(Hq, Hkv, ng, 1)
        assert len(groups) <= max(1, min(ng, Hkv))
        G = Hq // Hkv
        kv_seen, q_seen = [], []
        for ka, kb, qa, qb, with_kv in groups:
            assert kb > ka and (qa, qb) == (ka * G, kb * G) and with_kv
            kv_seen += list(range(ka, kb))
            q_seen += list(range(qa, qb))
        assert kv_seen == list(range(Hkv)) and q_seen == list(range(Hq))


def test_split_query_heads_keeps_coverage_and_kv_ownership():
    # the first and the last KV head are cut by query heads, the ones in between stay whole
    g = sab.host_forward_plan(32, 8, 8, 2)
    assert [x[2:4] for x in g] == [(0, 2), (2, 4)] + [(4 * i, 4 * i + 4) for i in range(1, 7)] + \
        [(28, 30), (30, 32)]
    assert [x[4] for x in g] == [True, False] + [True] * 6 + [True, False]   # K/V with the first part
    assert all(kb - ka == 1 for ka, kb, *_ in g)
    g = sab.host_forward_plan(32, 8, 8, 4)
    assert len(g) == 14 and [x[2:4] for x in g][-4:] == [(28, 29), (29, 30), (30, 31), (31, 32)]
    assert sab.host_forward_plan(4, 1, 1, 2) == [(0, 1, 0, 2, True), (0, 1, 2, 4, False)]
    # ranges with several KV heads, or an odd number of query heads per KV head, stay whole
    assert sab.host_forward_plan(8, 4, 2, 2) == [(0, 2, 0, 4, True), (2, 4, 4, 8, True)]
    assert sab.host_forward_plan(3, 1, 1, 2) == [(0, 1, 0, 3, True)]


def test_head_groups_rejects_bad_head_counts():
    with pytest.raises(ValueError):
        sab.host_forward_plan(10, 4, 2, 1)
    with pytest.raises(ValueError):
        sab.host_forward_plan(0, 1, 1, 1)


def test_host_forward_rejects_bad_arguments_before_any_cuda_call():
    import ctypes
    lib = sab.load_library()
    p = sab.SaProblem(B=1, Hq=4, Hkv=2, n=64, d=64, w=8, dtype=sab.BF16, flags=sab.CAUSAL)
    need = sab.host_forward_ws_bytes(1, 4, 2, 64, 64)
    assert need >= (3 * 4 + 2 * 2) * 64 * 64 * 2       # q, y, scratch + k, v
    fake = ctypes.c_void_p(0x10000)
    args = lambda ws, nbytes: (ctypes.byref(p), fake, fake, fake, fake, fake, 1, 0, 2, 1, ws,
                               nbytes, None)
    assert lib.sa_swa_gated_forward_host(*args(None, need)) == 1
    assert lib.sa_swa_gated_forward_host(*args(ctypes.c_void_p(0x10010), need)) == 1   # alignment
    assert lib.sa_swa_gated_forward_host(*args(fake, need - 1)) == 3


# the workspace as the library sizes it for the calls to come: with room of its own for key lists that do
# not fit beside the rest
@pytest.mark.parametrize("B,Hq,Hkv,n,d,w,extra", [
    (1, 2, 1, 32768, 64, 2048, True), (1, 4, 2, 33000, 64, 4000, True), (2, 2, 1, 33001, 64, 2000, True),
    (1, 4, 2, 33100, 64, 2000, False), (1, 2, 1, 32768, 64, 512, False), (1, 2, 2, 32768, 64, 2048, False),
])
def test_workspace_has_room_for_the_key_lists(B, Hq, Hkv, n, d, w, extra):
    import ctypes
    p = sab.SaProblem(B=B, Hq=Hq, Hkv=Hkv, n=n, d=d, w=w, dtype=sab.BF16, flags=sab.CAUSAL)
    sab.load_library().sa_problem_set_contiguous(ctypes.byref(p))
    need = sab.load_library().sa_host_forward_ws_bytes(ctypes.byref(p))
    least = sab.host_forward_ws_bytes(B, Hq, Hkv, n, d)
    assert sab.host_forward_ws_bytes(B, Hq, Hkv, n, d, w=w, flags=sab.CAUSAL) == need
    assert (need > least) == extra
    if extra:
        assert need - least == sab.sa_workspace_bytes(p, sab.OP_KEY_LISTS)


# what the call makes of a problem: every head of every sequence once, K and V with the first piece that
# reads them; many sequences with many groups, none, and more than there are events for
@pytest.mark.parametrize("B,Hq,Hkv,n,d,n_groups,q_parts", [
    (300, 8, 8, 683, 64, 300, 2), (300, 8, 8, 683, 64, 1000, 1), (16, 64, 32, 4096, 128, 512, 2),
    (1, 8, 1, 9600, 64, 1, 2), (1, 16, 2, 38000, 64, 256, 8), (8, 8, 2, 4096, 64, 0, 2),
    (8, 8, 2, 4096, 64, -1, 2), (300, 2, 2, 20000, 64, -5, 1),
])
def test_pieces_cover_every_head_of_every_sequence_once(B, Hq, Hkv, n, d, n_groups, q_parts):
    pieces = sab.host_forward_pieces(B, Hq, Hkv, n, d, sab.BF16, n_groups, q_parts)
    assert 1 <= len(pieces) <= 256
    if q_parts == 1:
        assert len(pieces) <= max(1, n_groups)
    q_seen, kv_seen = set(), set()
    for ka, kb, qa, qb, with_kv, b0, b1 in pieces:
        G = Hq // Hkv
        assert ka * G <= qa < qb <= kb * G and b0 < b1
        if with_kv:
            new = {(b, h) for b in range(b0, b1) for h in range(ka, kb)}
            assert not new & kv_seen
            kv_seen |= new
        assert all((b, h) in kv_seen for b in range(b0, b1) for h in range(ka, kb))
        new = {(b, h) for b in range(b0, b1) for h in range(qa, qb)}
        assert not new & q_seen
        q_seen |= new
    assert len(q_seen) == B * Hq and len(kv_seen) == B * Hkv
    if n_groups < 1 and q_parts == 1:
        assert len(pieces) == 1


def test_what_the_heads_alone_refuse_stays_refused():
    with pytest.raises(ValueError):
        sab.host_forward_pieces(1, 300, 300, 64, 64, n_groups=300)      # more pieces than 256
    with pytest.raises(ValueError):
        sab.host_forward_pieces(1, 10, 4, 64, 64)
    with pytest.raises(sab.SaError):
        sab.host_forward_pieces(0, 8, 4, 64, 64)


# Input enough for the pieces asked for (2 MB each): two sequences, then ranges of their heads; heads
# alone; and the first and last KV head cut by query heads, whose later part finds K and V on the GPU
# (half of 8 heads' 75 row tiles each still fill it).
@pytest.mark.gpu
@pytest.mark.parametrize("B,Hq,Hkv,n,n_groups,q_parts,pieces", [
    (2, 8, 4, 2100, 1, 1, 1), (2, 8, 4, 2100, 3, 2, 2), (2, 8, 4, 2100, 4, 2, 4), (2, 8, 4, 2100, 4, 1, 4),
    (1, 8, 4, 4200, 3, 2, 3), (1, 8, 4, 4200, 4, 1, 4),
    (1, 8, 1, 9600, 1, 2, 2), (1, 16, 2, 9600, 2, 2, 4), (1, 8, 1, 9600, 1, 4, 1),
])
def test_pipelined_forward_equals_single_call(B, Hq, Hkv, n, n_groups, q_parts, pieces):
    from paper_2604_00754_b200 import binding as sa
    d, w = 64, 256
    g = torch.Generator().manual_seed(11)
    q = torch.randn(B, Hq, n, d, generator=g).bfloat16().pin_memory()
    k = torch.randn(B, Hkv, n, d, generator=g).bfloat16().pin_memory()
    v = torch.randn(B, Hkv, n, d, generator=g).bfloat16().pin_memory()
    lg = torch.randn(2, Hq, generator=g).pin_memory()
    hy = torch.empty_like(q).pin_memory()
    hf = host.HostForward(B, Hq, Hkv, n, d, w, n_groups=n_groups, q_parts=q_parts)
    assert len(hf.pieces) == pieces
    dev = [t.cuda() for t in (q, k, v)]
    for layer in (2, 3):                   # another layer index draws another permutation
        launches = sa.launch_count()
        hf.forward(q, k, v, lg, hy, seed=5, layer=layer)
        assert sa.launch_count() - launches == 1 + 2 * pieces
        torch.cuda.synchronize()
        perm, inv = sa.sa_make_perm(5, layer, B, n)
        ref = sa.sa_swa_gated_forward(*dev, perm, inv, lg.cuda(), w)
        assert sa.sa_read_status() == 0
        assert torch.equal(hy, ref.cpu())


# more groups than events, and none: two launches per piece and one for the permutation
@pytest.mark.gpu
@pytest.mark.parametrize("B,n,n_groups", [(300, 683, 300), (4, 2100, -1)])
def test_any_number_of_groups(B, n, n_groups):
    from paper_2604_00754_b200 import binding as sa
    g = torch.Generator(device="cuda").manual_seed(n)
    dev = [torch.randn(B, 8, n, 64, generator=g, device="cuda").bfloat16() for _ in range(3)]
    lg = torch.randn(2, 8, generator=g, device="cuda")
    q, k, v, hlg = (torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t) for t in dev + [lg])
    hy = torch.empty(q.shape, dtype=q.dtype, pin_memory=True)
    hf = host.HostForward(B, 8, 8, n, 64, 32, n_groups=n_groups)
    launches = sa.launch_count()
    hf.forward(q, k, v, hlg, hy, seed=5, layer=2)
    assert sa.launch_count() - launches == 1 + 2 * len(hf.pieces)
    torch.cuda.synchronize()
    perm, inv = sa.sa_make_perm(5, 2, B, n)
    ref = sa.sa_swa_gated_forward(*dev, perm, inv, lg, 32)
    assert sa.sa_read_status() == 0
    assert torch.equal(hy, ref.cpu())

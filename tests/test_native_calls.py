"""The C++ entry of the per-layer calls: what it refuses, and how it shares the interpreter."""
import pytest
import torch

from paper_2604_00754_b200 import binding as sa

B, H, n, d, w = 2, 3, 16, 64, 5


# Rows of a packed projection and heads that are expanded: strides that no fresh tensor has.  With
# one set of strides for both, a kernel would write outside the output, so the call is refused
# (host tensors: nothing can be launched on them, with or without the check).
def _packed():
    return torch.zeros(B, 3 * H, n, d).bfloat16()[:, :H]


def _expanded():
    return torch.zeros(B, 1, n, d).bfloat16().expand(B, H, n, d)


@pytest.mark.parametrize("make", [_packed, _expanded])
@pytest.mark.parametrize("call", ["forward", "gated", "gated_saving", "backward_q", "backward_k",
                                  "rope", "gated_rope"])
def test_outputs_that_cannot_have_the_layout_are_refused(make, call):
    perm = torch.arange(n, dtype=torch.int32).expand(B, n).contiguous()
    odd, plain = make(), torch.zeros(B, H, n, d).bfloat16()
    assert torch.empty_like(odd).stride() != odd.stride()
    lg, lse = torch.zeros(2, H), torch.zeros(B, H, n)
    with pytest.raises(ValueError, match="layout"):
        if call == "forward":
            sa.sa_forward(odd, plain, plain, perm, perm, w)
        elif call.startswith("gated"):
            sa.sa_swa_gated_forward(odd, plain, plain, perm, perm, lg, w,
                                    save_for_bwd=call == "gated_saving")
        elif call == "rope":
            sa.sa_forward_rope(odd, plain, plain, perm, perm, lse, lse, w)
        elif call == "gated_rope":
            sa.sa_swa_gated_forward_rope(odd, plain, plain, perm, perm, lse, lse, lg, w)
        else:
            q, k = (odd, plain) if call == "backward_q" else (plain, odd)
            sa.sa_backward(q, k, k, perm, perm, lg, q, q, lse, lse, q, w)


# Numbers are taken as the Python calls took them: whole extents, and whatever float() takes.
@pytest.mark.parametrize("B, n", [(2.0, 16), (2, 16.5), ("2", 16)])
def test_extents_are_whole_numbers(B, n):
    perm, ws = torch.zeros(2, 16, dtype=torch.int32), torch.zeros(1 << 16, dtype=torch.uint8)
    with pytest.raises(TypeError):
        sa.sa_make_perm(1, 0, B, n, perm=perm, inv=perm.clone(), ws=ws)


@pytest.mark.gpu
def test_scale_is_what_float_takes():
    q = torch.randn(1, 1, 64, 64, device="cuda").bfloat16()
    perm, inv = sa.sa_make_perm(1, 0, 1, 64)
    want = sa.sa_forward(q, q, q, perm, inv, 8, scale=0.25)
    for scale in ("0.25", torch.tensor(0.25), 1 / 4):
        assert torch.equal(sa.sa_forward(q, q, q, perm, inv, 8, scale=scale), want)
    with pytest.raises(TypeError):
        sa.sa_forward(q, q, q, perm, inv, 8, scale=None)


# A launch waits where the device's queue is full (behind a kernel that runs for half a second here):
# the other threads of the interpreter go on meanwhile.
@pytest.mark.gpu
@pytest.mark.parametrize("call", ["make_perm", "forward", "gated", "backward"])
def test_a_waiting_launch_does_not_stop_other_threads(call):
    import threading
    import time
    q, y = (torch.zeros(1, 1, 64, 64, device="cuda").bfloat16() for _ in range(2))
    perm, inv = sa.sa_make_perm(1, 0, 1, 64)
    ws = torch.empty(1 << 20, dtype=torch.uint8, device="cuda")
    lg, lse = torch.zeros(2, 1, device="cuda"), torch.zeros(1, 1, 64, device="cuda")
    dgate = torch.empty_like(lg)
    grads = dict(dq=torch.empty_like(q), dk=torch.empty_like(q), dv=torch.empty_like(q), dgate=dgate)
    one = {"make_perm": lambda: sa.sa_make_perm(1, 0, 1, 64, perm=perm, inv=inv, ws=ws),
           "forward": lambda: sa.sa_forward(q, q, q, perm, inv, 8, y=y),
           "gated": lambda: sa.sa_swa_gated_forward(q, q, q, perm, inv, lg, 8, out=dict(y=y)),
           "backward": lambda: sa.sa_backward(q, q, q, perm, inv, lg, y, y, lse, lse, q, 8, ws=ws,
                                              out=grads)}[call]
    one()
    torch.cuda.synchronize()
    took = []

    def enqueue():
        t0 = time.perf_counter()
        for _ in range(3000):
            one()
        took.append(time.perf_counter() - t0)

    torch.cuda._sleep(1000000000)
    thread, gap = threading.Thread(target=enqueue), 0.0
    last = time.perf_counter()
    thread.start()
    while thread.is_alive():
        time.sleep(0.001)
        now = time.perf_counter()
        gap, last = max(gap, now - last), now
    thread.join()
    torch.cuda.synchronize()
    assert sa.sa_read_status() == 0
    assert took[0] > 0.3 and gap < 0.15, (took[0], gap)


# A launch that fails (here into a graph capture that a synchronisation has spoiled) is told by its own
# call and not once more by the next one.  In a process of its own: torch keeps the spoiled capture.
SPOILED = """
import sys, torch
sys.path.insert(0, sys.argv[1])
from paper_2604_00754_b200 import binding as sa
lib = sa.load_library()
t = [torch.empty(64, dtype=torch.int32, device="cuda") for _ in range(2)]
ws = torch.empty(1 << 16, dtype=torch.uint8, device="cuda")
draw = lambda s: lib.sa_make_perm(1, 0, 1, 64, t[0].data_ptr(), t[1].data_ptr(), ws.data_ptr(),
                                  ws.numel(), s.cuda_stream)
side, main = torch.cuda.Stream(), torch.cuda.current_stream()
assert draw(main) == 0
torch.cuda.synchronize()
with torch.cuda.stream(side):
    graph = torch.cuda.CUDAGraph()
    graph.capture_begin()
    codes = [lib.sa_read_status(side.cuda_stream), draw(side)]
    try:
        graph.capture_end()
    except RuntimeError:
        pass
codes.append(draw(main))
print(codes, lib.sa_read_status(main.cuda_stream))
"""


@pytest.mark.gpu
def test_a_failed_launch_is_told_once():
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = subprocess.run([sys.executable, "-c", SPOILED, root], capture_output=True, text=True, timeout=300)
    assert out.stdout.strip().endswith("[4, 4, 0] 0"), out.stdout + out.stderr

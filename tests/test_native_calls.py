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

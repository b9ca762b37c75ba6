"""Launches and algorithmic bytes that fhe_profile_end reports for a key switch and for a rotation key, on a ring of
single-pass transforms (one launch per transform, every row swept once)."""
import pytest

from tests.gpu_common import gpu_ctx

pytestmark = pytest.mark.gpu


def test_rotation_counts_its_rows_and_the_copies_of_the_first_transform():
    ctx = gpu_ctx("t10", 3, [1])
    level = ctx.top
    l1, alpha, n = level + 1, ctx.alpha, ctx.n
    a, out = ctx.empty_ct(), ctx.empty_ct()
    ctx.profile_begin()
    ctx.rotate(a, out, 1, level, 1)
    st = ctx.profile_end()
    digits = -(-l1 // alpha)
    raised = sum(l1 + alpha - min(alpha, l1 - j * alpha) for j in range(digits))
    inv_launches, _, inv_bytes, _ = st["ntt_inverse"]
    fwd_launches, _, fwd_bytes, _ = st["ntt_forward"]
    assert (inv_launches, fwd_launches) == (2, 2)
    assert inv_bytes == 16.0 * n * (l1 + 2 * alpha) + 8.0 * n * l1      # the digits' own limbs are stored beside
    assert fwd_bytes == 16.0 * n * (raised + 2 * l1)


def test_a_rotation_key_counts_every_launch():
    ctx = gpu_ctx("t10", 3)
    digits = -(-(ctx.top + 1) // ctx.alpha)
    ctx.profile_begin()
    ctx.add_rotation_keys([5])
    assert ctx.profile_end()["other"][0] == 1 + 2 * digits              # automorphism; key halves and storing per digit

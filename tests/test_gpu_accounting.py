"""Launches that fhe_profile_end reports for a rotation key."""
import pytest

from tests.gpu_common import gpu_ctx

pytestmark = pytest.mark.gpu


def test_a_rotation_key_counts_every_launch():
    ctx = gpu_ctx("t10", 3)
    digits = -(-(ctx.top + 1) // ctx.alpha)
    ctx.profile_begin()
    ctx.add_rotation_keys([5])
    assert ctx.profile_end()["other"][0] == 1 + 2 * digits              # automorphism; key halves and storing per digit

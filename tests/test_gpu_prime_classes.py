"""Every arithmetic of the transforms (near 50-bit, near 60-bit and any other primes) in single-pass
and two-pass rings, and base conversions from one to seven source limbs, bit for bit against the oracle;
transforms of residues at the ends of their range."""
import numpy as np
import pytest

from oracle import ckks
from paper_2509_03024_gb300 import capi
from tests.gpu_common import assert_ct_equal, built, ct_slice, to_coeff, torch

pytestmark = pytest.mark.gpu

# log_n, data prime bits, special prime bits, log_scale
RINGS = {
    "n10_mixed": (10, (61, 55, 50, 30), (61,), 30),
    "n11_near60": (11, (60, 50, 60), (50, 60), 40),
    "n9_seven_sources": (9, (50,) * 7, (60,) * 6, 40),      # fused ModDown-rescale converts from 7 limbs
    "n12_five_sources": (12, (60, 58, 50, 50, 40, 50), (61,) * 4 + (60,), 30),
    "n14": (14, (50, 60, 45, 50), (60, 61), 40),
    "n14_three_sources": (14, (50, 50, 60, 41), (60, 60, 57), 35),
}


def _pair(name, steps):
    log_n, data, special, scale = RINGS[name]
    built()
    ctx = capi.Context(log_n, data, special, scale)
    ctx.keygen(5, steps)
    he = ckks.Ckks(ckks.Params(log_n, data, special, scale))
    he.keygen(5, steps)
    return ctx, he


@pytest.mark.parametrize("name", sorted(RINGS))
def test_key_switch_and_rescale_bit_exact(name):
    steps = [1, 2, 3]
    ctx, he = _pair(name, steps)
    a = ctx.empty_ct(2)
    z = np.zeros(ctx.slots)
    z[:40] = np.random.default_rng(3).uniform(-1, 1, 40)
    for i in range(2):
        ctx.encrypt(np.roll(z, i), ctx.top, 90 + i, ct_slice(ctx, a, i))
    A, B = ct_slice(ctx, a, 0), ct_slice(ctx, a, 1)
    oa, ob = he.encrypt(z, he.prm.top, 90), he.encrypt(np.roll(z, 1), he.prm.top, 91)
    for level in (ctx.top, 1):
        xa, xb = he.drop(oa, level), he.drop(ob, level)
        out = ctx.empty_ct()
        ctx.rotate(A, out, 1, level, 3)
        assert_ct_equal(to_coeff(ctx, out, level)[0], he.rotate(xa, 3), f"rotate at {level}")
        ctx.mul_relin_rescale(A, B, out, 1, level)
        assert_ct_equal(to_coeff(ctx, out, level - 1)[0], he.relin_rescale(he.tensor(xa, xb)), f"product at {level}")
        ctx.rescale(A, out, 1, level)
        assert_ct_equal(to_coeff(ctx, out, level - 1)[0], he.rescale(xa), f"rescale at {level}")


@pytest.mark.parametrize("name", sorted(RINGS))
@pytest.mark.parametrize("variant", ["r16b4", "r8b4", "r32b4", "r16b3"])
def test_transform_of_extreme_residues(name, variant):
    """All-zero, all q - 1, alternating and random residues come back from forward and inverse
    transforms in either order; the transform of the constant q - 1 is q - 1 everywhere."""
    log_n, data, special, scale = RINGS[name]
    built()
    ctx = capi.Context(log_n, data, special, scale)
    ctx.set_variant("ntt", variant)
    n, L1 = ctx.n, ctx.top + 1
    rng = np.random.default_rng(8)
    rows = np.zeros((5, L1, n), dtype=np.uint64)
    for i, q in enumerate(ctx.primes[:L1]):
        rows[1, i] = q - 1
        rows[2, i, ::2] = q - 1
        rows[3, i] = rng.integers(0, q, n, dtype=np.uint64)
        rows[4, i, 0] = q - 1                              # the constant polynomial -1
    base = torch.from_numpy(rows.view(np.int64)).cuda()
    t = base.clone()
    ctx.ntt_forward(t, 5, L1)
    ev = t.cpu().numpy().view(np.uint64)
    for i, q in enumerate(ctx.primes[:L1]):
        assert (ev[0, i] == 0).all() and (ev[4, i] == q - 1).all() and (ev[:, i] < q).all()
    ctx.ntt_inverse(t, 5, L1)
    assert torch.equal(t, base)
    ctx.ntt_inverse(t, 5, L1)
    ctx.ntt_forward(t, 5, L1)
    assert torch.equal(t, base)

"""Residues at the ends of their range through every tile shape of the two-pass transforms, in launches large
enough that the shape asked for is the one that runs (16 residues per thread; smaller launches take 8 whatever
the choice): plain transforms, and the fused passes of rotations, products and rescales, for near 50-bit, near
60-bit and other primes in one ring."""
import numpy as np
import pytest

from oracle import ckks
from paper_2509_03024_gb300 import capi
from tests.gpu_common import assert_ct_equal, built, ct_slice, to_coeff, torch

pytestmark = pytest.mark.gpu

RINGS = {"mixed": ((50, 60, 61, 45), (60, 61)), "unreduced57": ((57, 57, 58, 57), (57, 57))}
SCALE = 40
rings = pytest.mark.parametrize("ring", sorted(RINGS))


def _line(ctx):
    """First number of rows whose launch gives every SM 512 threads of 16 residues."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return -(-sms * 512 * 16 // ctx.n)


def _patterns(ctx, polys):
    """[polys][limbs][N]: all q - 1; q - 1 at even, at odd places; in the lower, in the upper half; q - 1 once; random."""
    limbs, n = ctx.top + 1, ctx.n
    rng = np.random.default_rng(4)
    a = np.zeros((polys, limbs, n), dtype=np.uint64)
    for i, q in enumerate(ctx.primes[:limbs]):
        for t in range(polys):
            k = t % 7
            where = (slice(None), slice(0, n, 2), slice(1, n, 2), slice(0, n // 2), slice(n // 2, n), slice(0, 1))
            if k < 6:
                a[t, i, where[k]] = q - 1
            else:
                a[t, i] = rng.integers(0, q, n, dtype=np.uint64)
    return torch.from_numpy(a.view(np.int64).reshape(-1)).cuda()


@rings
@pytest.mark.parametrize("log_n", [14, 15, 16])
def test_plain_tile_shapes(log_n, ring):
    built()
    ctx = capi.Context(log_n, *RINGS[ring], SCALE)
    limbs = ctx.top + 1
    polys = -(-_line(ctx) // limbs) + 7
    w = limbs * ctx.n
    base = _patterns(ctx, polys)
    fwd, inv = base.clone(), base.clone()
    for t in range(polys):                                   # one polynomial a launch: 8 residues per thread
        ctx.ntt_forward(fwd[t * w:(t + 1) * w], 1, limbs)
        ctx.ntt_inverse(inv[t * w:(t + 1) * w], 1, limbs)
    for i, q in enumerate(ctx.primes[:limbs]):               # the constant q - 1 transforms to q - 1 everywhere
        assert (fwd.view(polys, limbs, ctx.n)[5, i] == q - 1).all()
        v = fwd.view(polys, limbs, ctx.n)[:, i].cpu().numpy().view(np.uint64)
        assert (v < q).all()
    for v in ("r16b4", "r8b4", "r32b4", "r16b3"):
        ctx.set_variant("ntt", v)
        x = base.clone()
        ctx.ntt_forward(x, polys, limbs)
        assert torch.equal(x, fwd), v
        ctx.ntt_inverse(x, polys, limbs)
        assert torch.equal(x, base), v
        ctx.ntt_inverse(x, polys, limbs)
        assert torch.equal(x, inv), v
        ctx.ntt_forward(x, polys, limbs)
        assert torch.equal(x, base), v


@rings
@pytest.mark.parametrize("log_n", [14, 15, 16])
def test_fused_tile_shapes(log_n, ring):
    built()
    ctx = capi.Context(log_n, *RINGS[ring], SCALE)
    ctx.keygen(6, [3])
    count, level = -(-_line(ctx) // 2) + 3, ctx.top          # the smallest launch has two rows per ciphertext
    a = _patterns(ctx, 2 * count)
    b = a.view(2 * count, -1).flip(0).contiguous().view(-1)  # the same polynomials in the other order
    ops = {"rotate": lambda x, y, o, n: ctx.rotate(x, o, n, level, 3),
           "product": lambda x, y, o, n: ctx.mul_relin_rescale(x, y, o, n, level),
           "rescale": lambda x, y, o, n: ctx.rescale(x, o, n, level)}
    picks = list(range(0, count, max(1, count // 6)))
    ref = {}
    for name, op in ops.items():
        for t in picks:
            one = ctx.empty_ct()
            op(ct_slice(ctx, a, t), ct_slice(ctx, b, t), one, 1)
            ref[name, t] = one
        for v in ("r16", "r8", "r8x"):
            ctx.set_variant("ks_pass", v)
            out = ctx.empty_ct(count)
            op(a, b, out, count)
            for t in picks:
                assert torch.equal(ct_slice(ctx, out, t), ref[name, t]), (name, v, t)
    if log_n == 14:
        he = ckks.Ckks(ckks.Params(log_n, *RINGS[ring], SCALE))
        he.keygen(6, [3])
        for t in picks[:3]:
            oa, ob = (ckks.Ciphertext(to_coeff(ctx, ct_slice(ctx, x, t), level)[0], level) for x in (a, b))
            got = {k: to_coeff(ctx, ref[k, t], level - (k != "rotate"))[0] for k in ops}
            assert_ct_equal(got["rotate"], he.rotate(oa, 3), "rotate")
            assert_ct_equal(got["product"], he.relin_rescale(he.tensor(oa, ob)), "product")
            assert_ct_equal(got["rescale"], he.rescale(oa), "rescale")

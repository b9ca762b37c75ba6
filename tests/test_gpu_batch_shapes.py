"""A large batch (16 residues per thread, every tile shape) gives the bits of the same items one by one (8
residues per thread, checked against the oracle elsewhere): transforms, rotations, products and rescales on
each two-pass ring, with batch sizes on both sides of the line between the two."""
import numpy as np
import pytest

from paper_2509_03024_gb300 import capi
from tests.gpu_common import built, ct_slice, torch

pytestmark = pytest.mark.gpu

RINGS = {12: ((60, 40, 50, 40), (60,), 30), 13: ((50, 40, 60), (60,), 40), 14: ((50, 50, 50), (60,), 50),
         15: ((50, 50, 50), (60, 60), 50), 16: ((50, 50, 50), (60,), 50)}


def _ctx(log_n):
    built()
    ctx = capi.Context(log_n, *RINGS[log_n])
    ctx.keygen(12, [5])
    return ctx


def _uniform(ctx, count, parts, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    out = torch.empty((count, parts, ctx.top + 1, ctx.n), dtype=torch.int64, device="cuda")
    for i in range(ctx.top + 1):
        out[:, :, i] = torch.randint(0, ctx.primes[i], (count, parts, ctx.n), generator=gen, device="cuda")
    return out.reshape(-1)


@pytest.mark.parametrize("log_n", sorted(RINGS))
def test_transforms(log_n):
    ctx = _ctx(log_n)
    limbs = ctx.top + 1
    line = -(-152 * 512 * 16 // (ctx.n * limbs))            # first count with 152 * 512 threads of 16 residues
    for count in (line - 1, line, line + 3):
        a = _uniform(ctx, count, 1, count)
        w = limbs * ctx.n
        one = a.clone()
        for t in range(count):
            ctx.ntt_forward(one[t * w:(t + 1) * w], 1, limbs)
        for v in ("r16b4", "r8b4", "r32b4", "r16b3"):
            ctx.set_variant("ntt", v)
            b = a.clone()
            ctx.ntt_forward(b, count, limbs)
            assert torch.equal(b, one), (count, v)
            ctx.ntt_inverse(b, count, limbs)
            assert torch.equal(b, a), (count, v)


@pytest.mark.parametrize("log_n", sorted(RINGS))
def test_key_switches_and_rescale(log_n):
    ctx = _ctx(log_n)
    count = -(-152 * 512 * 16 // ctx.n) + 1                 # enough for the launches of the fewest rows too
    level = ctx.top
    a, b = _uniform(ctx, count, 2, 1), _uniform(ctx, count, 2, 2)
    ops = {"rotate": lambda x, y, o, n: ctx.rotate(x, o, n, level, 5),
           "product": lambda x, y, o, n: ctx.mul_relin_rescale(x, y, o, n, level),
           "rescale": lambda x, y, o, n: ctx.rescale(x, o, n, level)}
    picks = sorted({0, 1, count // 2, count - 1})
    for name, op in ops.items():
        for v in ("r16", "r8", "r8x"):
            ctx.set_variant("ks_pass", v)
            out = ctx.empty_ct(count)
            op(a, b, out, count)
            for t in picks:
                one = ctx.empty_ct()
                op(ct_slice(ctx, a, t), ct_slice(ctx, b, t), one, 1)
                assert torch.equal(ct_slice(ctx, out, t), one), (name, v, t)

"""The ring of 2^12 between its two forms: plain transforms of the same extreme rows in one and in two passes
(launch sizes on both sides of each line), and fused passes in one."""
import numpy as np
import pytest

from paper_2509_03024_gb300 import capi
from tests.gpu_common import built, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [(50, 60, 61, 40)])
def test_both_forms_agree_at_the_lines(bits):
    built()
    ctx = capi.Context(12, bits, (60,), 40)
    n, limbs = ctx.n, 4
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(3)
    pat = np.zeros((4, limbs, n), dtype=np.uint64)
    for i, q in enumerate(ctx.primes[:limbs]):
        pat[0, i] = q - 1
        pat[1, i, ::2] = q - 1
        pat[2, i, n // 2:] = q - 1
        pat[3, i] = rng.integers(0, q, n, dtype=np.uint64)
    pat = torch.from_numpy(pat.view(np.int64)).cuda()
    one = {}
    for name, op in (("fwd", ctx.ntt_forward), ("inv", ctx.ntt_inverse)):
        one[name] = pat.clone()
        for t in range(4):                                   # four rows a launch: two passes
            op(one[name][t].view(-1), 1, limbs)
    for rows in (sms // 3, sms // 3 + 1, 4 * sms, 4 * sms + 4, 30 * sms):
        polys = -(-rows // limbs)
        for name, op in (("fwd", ctx.ntt_forward), ("inv", ctx.ntt_inverse)):
            x = pat.repeat(-(-polys // 4), 1, 1)[:polys].contiguous()
            want = one[name].repeat(-(-polys // 4), 1, 1)[:polys]
            op(x.view(-1), polys, limbs)
            assert torch.equal(x, want), (name, rows)


def test_fused_passes_are_one_launch_each():
    built()
    ctx = capi.Context(12, (50, 40, 40), (60,), 40)
    ctx.keygen(3, [1])
    for count in (1, 200):
        a, out = ctx.empty_ct(count), ctx.empty_ct(count)
        ctx.profile_begin()
        ctx.rotate(a, out, count, 2, 1)
        st = ctx.profile_end()
        assert st["ntt_forward"][0] == 2 and st["ntt_inverse"][0] == 2
        ctx.profile_begin()
        ctx.rescale(a, out, count, 2)
        st = ctx.profile_end()
        assert st["ntt_forward"][0] == 1 and st["ntt_inverse"][0] == 1

"""Client side against the oracle: decoding of any number of slots on every size of ring, encryption whose
ternary stream holds the one output the sampler rejects, and encodings of few and of many distinct values."""
import numpy as np
import pytest

from oracle import ckks
from paper_2509_03024_gb300 import capi
from tests.gpu_common import assert_ct_equal, built, to_coeff, torch

pytestmark = pytest.mark.gpu

GAMMA, M64 = 0x9E3779B97F4A7C15, (1 << 64) - 1


def _unmix64(y):
    """Inverse of the SplitMix64 output function."""
    def unshift(v, s):
        x = v
        for _ in range(0, 64, s):
            x = v ^ (x >> s)
        return x
    z = unshift(y, 31) * pow(0x94D049BB133111EB, -1, 1 << 64) & M64
    z = unshift(z, 27) * pow(0xBF58476D1CE4E5B9, -1, 1 << 64) & M64
    return unshift(z, 30)


@pytest.mark.parametrize("log_n", [9, 10, 13, 14, 15])
def test_decode_matches_direct_sum(log_n):
    """Slots of decrypted coefficients against the oracle's direct sum of N terms; both are float64 sums of
    |m_j| / Delta with rounding below (N + 64) 2^-53 of the sum of magnitudes."""
    built()
    ctx = capi.Context(log_n, (60, 40), (60,), 40)
    he = ckks.Ckks(ckks.Params(log_n, (60, 40), (60,), 40))
    ctx.keygen(3)
    he.keygen(3)
    z = np.random.default_rng(log_n).normal(0, 2, 60)
    for level in (1, 0):
        ct = ctx.empty_ct()
        ctx.encrypt(z, level, 17, ct)
        m = he.decrypt_coeffs(he.encrypt(z, level, 17))
        tol = (ctx.n + 64) * 2.0 ** -53 * float(sum(abs(int(v)) for v in m)) / 2.0 ** 40
        for count in (1, 33, ctx.slots if log_n < 14 else 257):
            got = ctx.decrypt(ct, level, count)
            assert got.shape == (count,)
            assert np.abs(got - he.enc.decode(m, count=count)).max() <= tol
        full = ctx.decrypt(ct, level)
        assert (full[:33] == ctx.decrypt(ct, level, 33)).all()


@pytest.mark.parametrize("bits", [(60, 40), (61, 61), (20, 50)])
@pytest.mark.parametrize("log_n", [11, 12, 16])
def test_decode_by_direct_sums_and_by_transform(log_n, bits):
    """The last ring decoded by direct sums, the first by a transform and the largest: two launches each, any number of
    slots a prefix of all, within the rounding of float64 sums of the oracle's, for extreme pairs of primes."""
    built()
    scale = min(bits[0] - 8, 40)
    ctx = capi.Context(log_n, bits, (61,), scale)
    he = ckks.Ckks(ckks.Params(log_n, bits, (61,), scale))
    ctx.keygen(3)
    he.keygen(3)
    z = np.random.default_rng(log_n).normal(0, 2, 40)
    for level in (1, 0):
        ct = ctx.empty_ct()
        ctx.encrypt(z, level, 17, ct)
        m = he.decrypt_coeffs(he.encrypt(z, level, 17))
        tol = (ctx.n + 64) * 2.0 ** -53 * float(sum(abs(int(v)) for v in m)) / 2.0 ** scale
        ctx.profile_begin()
        full = ctx.decrypt(ct, level)
        assert ctx.profile_end()["encode"][0] == 2
        count = 2048 if log_n < 16 else 97
        assert np.abs(full[:count] - he.enc.decode(m, count=min(count, ctx.slots))).max() <= tol
        for count in (1, 33, 700):
            assert (full[:count] == ctx.decrypt(ct, level, count)).all()


@pytest.mark.parametrize("at", [1, 2, 700, 1024, 1025])
def test_encryption_past_a_rejected_ternary_draw(at):
    """A seed whose ternary stream of nonce 9 outputs 2^64 - 1 (rejected) at counter `at` of N = 1024."""
    built()
    h = (_unmix64(M64) - at * GAMMA) & M64               # state before the stream: mix64(h + at gamma) = 2^64 - 1
    for f in (0, 0, 9, 6):                               # limb, poly, object, purpose
        h = ((_unmix64(h) - GAMMA) & M64) ^ f
    data, special = (60, 40, 40), (60,)
    ctx = capi.Context(10, data, special, 40)
    ctx.keygen(h)
    he = ckks.Ckks(ckks.Params(10, data, special, 40))
    he.keygen(h)
    assert int(ckks.draws(ckks.stream_key(h, 6, 9), at - 1, 1)[0]) == M64
    ct = ctx.empty_ct()
    ctx.encrypt(np.ones(3), 2, 9, ct)
    assert_ct_equal(to_coeff(ctx, ct, 2)[0], he.encrypt(np.ones(3), 2, 9), "encrypt")


def test_encryption_with_the_rejected_state_as_stream_key():
    """The ternary stream of nonce 9 starts in the one state the sampler rejects: counters start at 1, so the
    stream holds no rejected output and nothing is skipped."""
    built()
    h = _unmix64(M64)
    for f in (0, 0, 9, 6):
        h = ((_unmix64(h) - GAMMA) & M64) ^ f
    data, special = (60, 40, 40), (60,)
    ctx = capi.Context(10, data, special, 40)
    ctx.keygen(h)
    he = ckks.Ckks(ckks.Params(10, data, special, 40))
    he.keygen(h)
    assert ckks.stream_key(h, 6, 9) == _unmix64(M64)
    ct = ctx.empty_ct()
    ctx.encrypt(np.ones(3), 2, 9, ct)
    assert_ct_equal(to_coeff(ctx, ct, 2)[0], he.encrypt(np.ones(3), 2, 9), "encrypt")


@pytest.mark.parametrize("log_n", [9, 11, 14])
@pytest.mark.parametrize("distinct,count", [(1, 1), (1, 200), (7, 56), (7, 55), (32, 256), (33, 250)])
def test_encode_few_and_many_distinct_values(log_n, distinct, count):
    """Both forms of the encoding (products tabulated per distinct value, or formed per term) and the
    rule between them give the oracle's integers."""
    built()
    ctx = capi.Context(log_n, (60, 40), (60,), 40)
    he = ckks.Ckks(ckks.Params(log_n, (60, 40), (60,), 40))
    rng = np.random.default_rng(distinct * 1000 + count)
    vals = rng.normal(0, 3, distinct)
    z = np.zeros(ctx.slots)
    slots = np.sort(rng.choice(ctx.slots, count, replace=False))
    z[slots] = vals[np.arange(count) % distinct]
    out = torch.zeros(ctx.n, dtype=torch.int64, device="cuda")
    ctx.encode(z, out)
    assert np.array_equal(out.cpu().numpy(), he.enc.encode(z))


@pytest.mark.parametrize("log_n,distinct,count,tabulated", [
    (9, 1, 256, True), (10, 1, 207, False), (10, 1, 208, True), (10, 5, 512, True), (12, 5, 243, False), (12, 5,
    244, True), (12, 16, 340, False), (12, 16, 342, True), (13, 1, 60, False), (14, 32, 512, True), (15, 1, 116,
    False), (15, 1, 117, True), (15, 16, 128, False), (15, 16, 192, True), (16, 1, 58, False), (16, 1, 59, True),
    (16, 33, 600, False)])
def test_products_are_tabulated_where_it_pays(log_n, distinct, count, tabulated):
    """Both sides of the rule's line: the launches it chooses, and the oracle's integers."""
    built()
    ctx = capi.Context(log_n, (60, 40), (60,), 40)
    he = ckks.Ckks(ckks.Params(log_n, (60, 40), (60,), 40))
    rng = np.random.default_rng(count)
    z = np.zeros(ctx.slots)
    z[np.sort(rng.choice(ctx.slots, count, replace=False))] = rng.normal(0, 3, distinct)[np.arange(count) % distinct]
    out = torch.zeros(ctx.n, dtype=torch.int64, device="cuda")
    ctx.profile_begin()
    ctx.encode(z, out)
    assert ctx.profile_end()["encode"][0] == (2 if tabulated else 1)
    assert np.array_equal(out.cpu().numpy(), he.enc.encode(z))

"""The one-drain tensor-core products (shorter operand of at most 512 limbs:
32-digit x blocks, one accumulator per tile, every block's Hankel matrices
resident) at the edges of their blocks, tiles and range, bit-exact against
the oracle."""
import numpy as np
import pytest

from helpers import to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bi():
    import paper_2607_28897_gb300 as m

    m.load()
    return m


def operands(na, nb, count):
    """Random rows, then rows that reach the accumulator bound (every digit
    +-128, with and without a carry digit), all ones, one and zero."""
    from paper_2607_28897_gb300 import inputs

    a, b = inputs.limbs(31 * na + nb, count, na), inputs.limbs(37 * nb + na + 1, count, nb)
    pats = (0x807F807F807F807F, 0x7F807F807F807F80, 0xFFFFFFFFFFFFFFFF, 1, 0)
    k = 0
    for x in pats:
        for y in pats[:3] if x else pats[:1]:
            a[k], b[k] = np.uint64(x), np.uint64(y)
            k += 1
    return a, b


@pytest.mark.parametrize("na,nb", [
    (64, 64), (65, 64), (80, 79), (127, 65), (128, 128), (129, 128), (160, 160), (256, 64),
    (240, 256), (255, 257), (257, 256), (333, 200), (511, 64), (511, 512), (512, 512),
    (513, 512), (512, 700), (1000, 128), (1024, 300), (1500, 512), (2000, 97), (4001, 130)])
def test_full_and_low(bi, orc, na, nb):
    a, b = operands(na, nb, 20)
    want = orc.batch_mul(a, b)
    assert np.array_equal(to_host(bi.mul(to_dev(a), to_dev(b))), want)
    for m in {1, min(na, nb), (na + nb) // 2 + 1, na + nb - 1}:
        got = to_host(bi.mul_lo(to_dev(a), to_dev(b), m))
        assert np.array_equal(got, want[:, :m]), m
    bi.check_timeout()


@pytest.mark.parametrize("n,count", [(64, 1300), (160, 1300), (256, 1300), (512, 700)])
def test_many_per_cta(bi, orc, n, count):
    """More products than resident CTAs: shared and tensor memory are reused;
    the patterns come first, last and between."""
    a, b = operands(n, n, count)
    a[-20:], b[-20:] = a[:20][::-1], b[:20][::-1]
    got = to_host(bi.mul(to_dev(a), to_dev(b)))
    assert np.array_equal(got, orc.batch_mul(a, b))
    bi.check_timeout()


@pytest.mark.parametrize("nu,nv", [(200, 130), (300, 200), (520, 260), (700, 300), (1024, 512),
                                   (1030, 513)])
def test_banded_in_division(bi, orc, nu, nv):
    """Band-mode products (columns dropped below a limb) inside step-batched
    divisions: quotients and remainders exact."""
    from paper_2607_28897_gb300 import inputs

    count = 40
    u, v = inputs.limbs(nu, count, nu, True), inputs.limbs(nv + 7, count, nv, True)
    u[0], v[0] = np.uint64(0xFFFFFFFFFFFFFFFF), np.uint64(0x7F807F807F807F80)
    u[1], v[1] = np.uint64(0x807F807F807F807F), np.uint64(0xFFFFFFFFFFFFFFFF)
    v[2] = 0
    v[2, -1] = 1
    q, r, st = bi.divmod(to_dev(u), to_dev(v))
    oq, orr, ost = orc.batch_divmod(u, v)
    assert np.array_equal(to_host(q), oq) and np.array_equal(to_host(r), orr)
    assert np.array_equal(st.cpu().numpy(), ost)
    bi.check_timeout()


@pytest.mark.parametrize("na,nb", [
    (513, 513), (520, 513), (515, 1024), (1024, 527), (528, 528), (544, 640), (600, 600),
    (513, 1500)])
def test_two_accumulators(bi, orc, na, nb):
    """Shorter operands just above one accumulator's bound, where even and odd
    blocks are summed apart: full and low products, more of them than CTAs."""
    count = 330
    a, b = operands(na, nb, count)
    a[-20:], b[-20:] = a[:20], b[:20]
    want = orc.batch_mul(a, b)
    assert np.array_equal(to_host(bi.mul(to_dev(a), to_dev(b))), want)
    for m in (min(na, nb), na + nb - 3):
        got = to_host(bi.mul_lo(to_dev(a), to_dev(b), m))
        assert np.array_equal(got, want[:, :m]), m
    bi.check_timeout()


@pytest.mark.parametrize("nu,nv", [(1024, 512), (1040, 520), (1200, 640), (1100, 512)])
def test_two_accumulators_banded(bi, orc, nu, nv):
    """The banded products of divisions with quotients of 513 to 700 limbs."""
    a, b = operands(nu, nv, 200)
    b[b[:, -1] == 0, -1] = 1
    q, r, st = bi.divmod(to_dev(a), to_dev(b))
    oq, orr, _ = orc.batch_divmod(a, b)
    assert not to_host(st).any()
    assert np.array_equal(to_host(q), oq) and np.array_equal(to_host(r), orr)
    bi.check_timeout()

"""The pipelined tensor-core products (builder, issuing and drain warps; 128-
and 64-digit x blocks) at the edges of their groups, tiles, buffers and
range, bit-exact against the oracle."""
import numpy as np
import pytest

from helpers import to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bi():
    import paper_2607_28897_gb300 as m

    m.load()
    return m


PATTERNS = (0x807F807F807F807F, 0x7F807F807F807F80, 0xFFFFFFFFFFFFFFFF, 1, 0)


def operands(na, nb, count):
    """Random rows and rows that reach the accumulator bound (every digit
    +-128), all ones, one and zero, in front."""
    from paper_2607_28897_gb300 import inputs

    a, b = inputs.limbs(41 * na + nb, count, na), inputs.limbs(43 * nb + na + 1, count, nb)
    for k in range(min(5, count - 1)):
        a[k], b[k] = np.uint64(PATTERNS[k]), np.uint64(PATTERNS[(k * k) % 4])
    return a, b


@pytest.mark.parametrize("na,nb", [
    (600, 600), (700, 513), (1000, 900), (1024, 1024), (1025, 1023), (1701, 1103), (2047, 2048),
    (2048, 2048), (2050, 2049), (2300, 700), (3000, 3100), (4096, 4096), (5000, 600), (600, 5000),
    (8192, 8192), (9000, 8999), (9900, 2000)])
def test_full_and_low(bi, orc, na, nb):
    a, b = operands(na, nb, 7)
    want = orc.batch_mul(a, b)
    assert np.array_equal(to_host(bi.mul(to_dev(a), to_dev(b))), want)
    for m in {min(na, nb) + 1, (na + nb) // 2 + 17, na + nb - 1}:
        got = to_host(bi.mul_lo(to_dev(a), to_dev(b), m))
        assert np.array_equal(got, want[:, :m]), m
    bi.check_timeout()


@pytest.mark.parametrize("na,nb,count", [(640, 600, 800), (1024, 1024, 620), (2048, 2048, 480),
                                         (1701, 1103, 470), (3000, 2100, 310)])
def test_across_products(bi, orc, na, nb, count):
    """Several products per CTA: operand buffers, stages and accumulators run
    on from one to the next, the patterns first, last and between."""
    a, b = operands(na, nb, count)
    a[-5:], b[-5:] = a[:5][::-1], b[:5][::-1]
    da, db = to_dev(a), to_dev(b)
    got = to_host(bi.mul(da, db))
    assert np.array_equal(got, orc.batch_mul(a, b))
    m = na + 3
    assert np.array_equal(to_host(bi.mul_lo(da, db, m)), got[:, :m])
    bi.check_timeout()


@pytest.mark.parametrize("nu,nv,count", [(2600, 1300, 200), (4100, 2050, 170), (6000, 4500, 160),
                                         (9000, 1500, 20)])
def test_banded_in_division(bi, orc, nu, nv, count):
    """Band-mode products inside step-batched divisions: quotients and
    remainders exact."""
    from paper_2607_28897_gb300 import inputs

    u, v = inputs.limbs(nu, count, nu, True), inputs.limbs(nv + 7, count, nv, True)
    u[0], v[0] = np.uint64(PATTERNS[2]), np.uint64(PATTERNS[1])
    u[1], v[1] = np.uint64(PATTERNS[0]), np.uint64(PATTERNS[2])
    v[2] = 0
    v[2, -1] = 1
    q, r, st = bi.divmod(to_dev(u), to_dev(v))
    pick = [0, 1, 2, 3, count // 2, count - 2, count - 1]
    oq, orr, ost = orc.batch_divmod(u[pick], v[pick])
    assert np.array_equal(to_host(q)[pick], oq) and np.array_equal(to_host(r)[pick], orr)
    assert np.array_equal(st.cpu().numpy()[pick], ost) and not st.any()
    # every instance: q v + r = u modulo B^nv (low products of their own)
    back = to_host(bi.mul_lo(q, to_dev(v), nv))
    s, _ = bi.add(to_dev(back), r)
    assert np.array_equal(to_host(s), u[:, :nv])
    bi.check_timeout()

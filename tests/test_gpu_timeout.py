"""The tensor-core products' device waits give up cleanly.  With an
injected timeout (a negative wait limit: each wait, once the MMAs it guards
have finished, runs out on a flag that nothing sets) a multiply and a
division report BIGINT_ETIMEOUT (bigint_check_timeout, the division's
per-instance status), the CTAs release their tensor memory, and after the
default limit is restored the next calls on the same device are bit-exact
against the oracle.  No fault is involved."""
import numpy as np
import pytest

from helpers import to_dev, to_host

pytestmark = pytest.mark.gpu


def test_wait_limit_timeout_then_recovery(orc):
    import torch

    import paper_2607_28897_gb300 as bi
    from paper_2607_28897_gb300 import inputs

    a, b = inputs.config_small(seed=9, n=512, count=4)  # 2^15-bit tensor-core products
    u, v = inputs.config_div(1024, 4, seed=10)  # division with tensor-core products
    assert bi.mul_variant_for(512, 512) == 12
    bi.check_timeout()  # nothing recorded before
    bi.set_wait_limit(-2000)
    try:
        bi.mul(to_dev(a), to_dev(b))
        with pytest.raises(bi.BigIntError) as e:
            bi.check_timeout()
        assert e.value.code == bi.ETIMEOUT
        q, r, st = bi.divmod(to_dev(u), to_dev(v))
        torch.cuda.synchronize()
        st = st.cpu().numpy()
        assert (st == bi.ETIMEOUT).all(), st
        assert set(np.unique(st)) <= {0, bi.ETIMEOUT}, st
        with pytest.raises(bi.BigIntError) as e:
            bi.check_timeout()
        assert e.value.code == bi.ETIMEOUT
        # an instance that finished before any wait gave up is still exact
        oq, orr, _ = orc.batch_divmod(u, v)
        ok = st == 0
        assert np.array_equal(to_host(q)[ok], oq[ok]) and np.array_equal(to_host(r)[ok], orr[ok])
    finally:
        bi.set_wait_limit(0)
    bi.check_timeout()  # the record was cleared by the reads above
    p = bi.mul(to_dev(a), to_dev(b))
    assert np.array_equal(to_host(p), orc.batch_mul(a, b))
    q, r, st = bi.divmod(to_dev(u), to_dev(v))
    oq, orr, ost = orc.batch_divmod(u, v)
    assert np.array_equal(to_host(q), oq) and np.array_equal(to_host(r), orr)
    assert not st.cpu().numpy().any()
    bi.check_timeout()


def test_pipeline_and_batch_give_up_then_recover(orc):
    """The same for the pipelined products (several per CTA, full ones and
    Poly's low ones with an addend) and the grouped products and divisions of
    a ragged batch."""
    import torch

    import paper_2607_28897_gb300 as bi
    from paper_2607_28897_gb300 import inputs

    n = 400  # more products than SMs
    a, b = (inputs.limbs(s, n, 2048, top_nonzero=True) for s in (31, 32))
    pa, pb = (inputs.limbs(s, n, 1024, top_nonzero=True) for s in (33, 34))
    ops, nin, nout = inputs.ragged_ops(35, 400, min_limbs=300, max_limbs=2000)
    pool = inputs.ragged_pool(36, ops, nin)
    da, db, dpa, dpb, dpool = (to_dev(x) for x in (a, b, pa, pb, pool))
    batch = bi.Batch(ops)
    out = torch.zeros(nout, dtype=torch.int64, device="cuda")
    st = torch.zeros(len(ops), dtype=torch.int32, device="cuda")

    def gave_up():
        with pytest.raises(bi.BigIntError) as e:
            bi.check_timeout()
        assert e.value.code == bi.ETIMEOUT

    bi.check_timeout()
    bi.set_wait_limit(-2000)
    try:
        bi.mul(da, db)
        gave_up()
        bi.poly(dpa, dpb)
        gave_up()
        batch.launch(dpool, out, st, mode=bi.BATCH_STEPS)
        gave_up()
        got = st.cpu().numpy()
        assert (got[ops["op"] >= 3] == bi.ETIMEOUT).all(), got
    finally:
        bi.set_wait_limit(0)
    bi.check_timeout()
    assert np.array_equal(to_host(bi.mul(da, db))[::40], orc.batch_mul(a[::40], b[::40]))
    got = to_host(bi.poly(dpa, dpb))
    for i in (0, 151, 152, n - 1):
        x, y = (int.from_bytes(v[i].tobytes(), "little") for v in (pa, pb))
        want = ((x * x + y) * (y * y + y) + x * y) % (1 << (64 * 1024))
        assert int.from_bytes(got[i].tobytes(), "little") == want, i
    batch.launch(dpool, out, st, mode=bi.BATCH_STEPS)
    got, status = to_host(out), st.cpu().numpy()
    for i in np.nonzero(ops["op"] >= 3)[0][::9]:
        o = ops[i]
        x, y = (int.from_bytes(pool[o[k]:o[k] + o[m]].tobytes(), "little")
                for k, m in (("a", "na"), ("b", "nb")))
        want = [(x * y, o["o1"], o["na"] + o["nb"])]
        if o["op"] == 4:
            want = [(x // y, o["o1"], o["na"] - o["nb"] + 1), (x % y, o["o2"], o["nb"])]
        assert status[i] == 0
        for value, at, size in want:
            assert int.from_bytes(got[at:at + size].tobytes(), "little") == value, i
    bi.check_timeout()

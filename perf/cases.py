"""The measured workload: batched big-integer arithmetic through the public
entry points of ``paper_2607_28897_gb300``.

Operands are unsigned integers as little-endian arrays of 64-bit limbs,
``(count, n)`` int64 tensors on the GPU.  The sizes follow the library's own
configurations: 2^15 .. 2^19-bit operands (512 .. 8192 limbs), operand arrays
of 2^32 bits, 2n-by-n-limb divisions, ragged mixed batches with sizes 2^U
bits (U uniform on [15, 19]), plus the smaller, unequal and odd sizes that
the entry points take.  Result buffers, workspaces and the plan of a ragged
batch are kept in the state, as a program that repeats a call keeps them.
Every result is an integer and has to agree bit for bit.
"""
from __future__ import annotations

import torch

import paper_2607_28897_gb300 as bi
from paper_2607_28897_gb300 import inputs


def listed():
    return [
        # A handful of products from one request, the small configuration's
        # 64 random and 8 carry-stress pairs: less than one wave of CTAs, so
        # launch and latency count.
        {"name": "mul_72x512", "op": "mul", "count": 72, "na": 512, "nb": 512},
        # The size sweep's 2^15-bit products: the throughput of the smallest
        # midsize operands.
        {"name": "mul_131072x512", "op": "mul", "count": 131072, "na": 512, "nb": 512},
        # Products of unequal odd-sized operands, as a ragged program meets
        # them once it has grouped equal shapes.
        {"name": "mul_16384x1701x1103", "op": "mul", "count": 16384, "na": 1701, "nb": 1103},
        # Products below the midsize range (10240 bits), the leaves of a
        # caller's own recursion: many at a time.
        {"name": "mul_65536x160", "op": "mul", "count": 65536, "na": 160, "nb": 160},
        # The sweep's largest products, 2^19 bits, in the sub-quadratic form.
        {"name": "kara_8192x8192", "op": "kara", "count": 8192, "na": 8192, "nb": 8192},
        # Addition at the sweep's largest size: HBM traffic only.
        {"name": "add_8192x8192", "op": "add", "count": 8192, "na": 8192, "nb": 8192},
        # Subtraction at an odd size: rows that start off a 16-byte boundary.
        {"name": "sub_40000x1537", "op": "sub", "count": 40000, "na": 1537, "nb": 1537},
        # The six-addition program on 2^17-bit operands.
        {"name": "chain_32768x2048", "op": "chain", "count": 32768, "na": 2048, "nb": 2048, "k": 6},
        # The polynomial program (four same-width products, three additions)
        # on 2^16-bit operands.
        {"name": "poly_16384x1024", "op": "poly", "count": 16384, "na": 1024, "nb": 1024},
        # The division configuration's smallest shape, 4096 at a time.
        {"name": "divmod_4096x1024x512", "op": "divmod", "count": 4096, "na": 1024, "nb": 512},
        # One 2^20-by-2^19-bit division, as a server answers a lone request:
        # a chain of dependent steps, latency only.
        {"name": "divmod_1x16384x8192", "op": "divmod", "count": 1, "na": 16384, "nb": 8192},
        # A ragged batch of mixed operations (40 % mul, 30 % add and sub,
        # 30 % divmod) on 2^15 .. 2^19 bits, its plan kept and replayed.
        {"name": "batch_20000", "op": "batch", "count": 20000, "ops_seed": 4},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    """One more case: the kinds above with sizes over their ranges."""
    op = rng.choice(["mul", "mul", "kara", "add", "sub", "chain", "poly", "divmod", "divmod",
                     "batch"])
    if op == "batch":
        return {"op": op, "count": _log_int(rng, 500, 20000), "ops_seed": rng.randrange(1000)}
    if op in ("add", "sub", "chain"):
        n = _log_int(rng, 64, 8192)
        if rng.random() < 0.5:
            n |= 1
        count = max(1, _log_int(rng, 1 << 14, 1 << 26) // n)
        case = {"op": op, "count": count, "na": n, "nb": n}
        if op == "chain":
            case["k"] = rng.randint(1, 12)
        return case
    if op == "divmod":
        nb = _log_int(rng, 64, 8192)
        na = nb + int(nb * rng.random()) if rng.random() < 0.5 else 2 * nb
        work = 2.0 ** rng.uniform(20, 31)  # limb products of the batch
        return {"op": op, "count": max(1, min(4096, int(work / (nb * nb)))), "na": na, "nb": nb}
    if op == "kara":
        na = nb = 8 * _log_int(rng, 256, 1024)
    else:
        na = _log_int(rng, 64, 8192)
        nb = na if op == "poly" or rng.random() < 0.5 else max(64, int(na * rng.uniform(0.3, 1.0)))
    work = 2.0 ** rng.uniform(24, 34)
    return {"op": op, "count": max(1, min(131072, int(work / (na * nb)))), "na": na, "nb": nb}


def _limbs(count, n, gen):
    """Uniform limbs with a nonzero top limb."""
    x = torch.randint(-2**63, 2**63 - 1, (count, n), dtype=torch.int64, device="cuda",
                      generator=gen)
    x[:, -1] |= 1
    return x


def _operands(case, seed):
    """The two operands of a uniform case.  Batches of 64 and more start with
    eight carry-stress pairs where the operands are equally long (all ones,
    one, zero, single-limb holes); every second divisor has bit 63 set, the
    others a top limb in [1, 2^32)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1000003 * seed + 17)
    count, na, nb = case["count"], case["na"], case["nb"]
    a, b = _limbs(count, na, gen), _limbs(count, nb, gen)
    if case["op"] == "divmod":
        b[0::2, -1] |= -2**63
        b[1::2, -1] = (b[1::2, -1] & 0xFFFFFFFF) | 1
    elif na == nb and count >= 64:
        sa, sb = inputs.stress_pairs(na)
        a[:8] = torch.from_numpy(sa.view("int64")).cuda()
        b[:8] = torch.from_numpy(sb.view("int64")).cuda()
    return a, b


def _bytes(n):
    return torch.empty(max(n, 256), dtype=torch.uint8, device="cuda")


def _empty(count, n, dtype=torch.int64):
    return torch.empty((count, n) if n else (count,), dtype=dtype, device="cuda")


def prepare(case, seed):
    op, count = case["op"], case["count"]
    if op == "batch":
        ops, n_in, n_out = inputs.ragged_ops(case["ops_seed"], count)
        gen = torch.Generator(device="cuda")
        gen.manual_seed(1000003 * seed + 17)
        pool = _limbs(1, n_in, gen).view(-1)
        tops = [ops["a"] + ops["na"] - 1, ops["b"] + ops["nb"] - 1]
        for t in tops:
            pool[torch.from_numpy(t.copy()).cuda()] |= 1
        return {"op": op, "plan": bi.Batch(ops), "a": pool,
                "out": torch.zeros(n_out, dtype=torch.int64, device="cuda"),
                "status": _empty(count, 0, torch.int32)}
    na, nb = case["na"], case["nb"]
    a, b = _operands(case, seed)
    s = {"op": op, "a": a, "b": b, "k": case.get("k", 0)}
    if op in ("add", "sub", "chain"):
        s["out"], s["flag"] = _empty(count, na), _empty(count, 0, torch.uint8)
    elif op == "mul":
        s["out"] = _empty(count, na + nb)
    elif op == "kara":
        s["out"] = _empty(count, na + nb)
        s["ws"] = _bytes(bi.mul_kara_workspace_bytes(count, na))
    elif op == "poly":
        s["out"] = _empty(count, na)
        s["ws"] = _bytes(bi.poly_workspace_bytes(count, na))
    else:
        s["q"], s["r"] = _empty(count, na - nb + 1), _empty(count, nb)
        s["status"] = _empty(count, 0, torch.int32)
        s["ws"] = _bytes(bi.divmod_workspace_bytes(count, na, nb))
    return s


def run(state):
    op = state["op"]
    if op == "mul":
        return bi.mul(state["a"], state["b"], out=state["out"])
    if op == "kara":
        return bi.mul_kara(state["a"], state["b"], out=state["out"], workspace=state["ws"])
    if op == "add":
        return bi.add(state["a"], state["b"], out=state["out"], carry=state["flag"])
    if op == "sub":
        return bi.sub(state["a"], state["b"], out=state["out"], borrow=state["flag"])
    if op == "chain":
        bi.add_chain(state["a"], state["b"], state["k"], out=state["out"], carry=state["flag"])
        return state["out"], state["flag"]
    if op == "poly":
        return bi.poly(state["a"], state["b"], out=state["out"], workspace=state["ws"])
    if op == "divmod":
        return bi.divmod(state["a"], state["b"], q=state["q"], r=state["r"],
                         status=state["status"], workspace=state["ws"])
    state["plan"].launch(state["a"], state["out"], state["status"], mode=bi.BATCH_STEPS)
    return state["out"], state["status"]


# Multiply-adds of 8-bit digits of one na-by-nb-limb product, as the digit
# convolution does them.
def _product(na, nb):
    return 64.0 * na * nb


def _division(na, nb):
    """A quotient of nq limbs: the Newton inverse (about nq^2), half of u w
    and half of q v."""
    nq = max(na - nb + 1, 1)
    return _product(nq, nb) + _product(nq, min(nq, nb))


def work(case):
    op, count = case["op"], case["count"]
    if op == "batch":
        ops, n_in, n_out = inputs.ragged_ops(case["ops_seed"], count)
        macs = 0.0
        for kind, na, nb in zip(ops["op"].tolist(), ops["na"].tolist(), ops["nb"].tolist()):
            if kind == bi.OP_MUL:
                macs += _product(na, nb)
            elif kind == bi.OP_DIVMOD:
                macs += _division(na, nb)
        return {"bytes": 8 * (n_in + n_out) + 4 * count, "flops": 2 * macs}
    na, nb = case["na"], case["nb"]
    if op in ("add", "sub", "chain"):
        return {"bytes": count * (24 * na + 1), "flops": count * na * case.get("k", 1)}
    if op == "mul":
        return {"bytes": count * 16 * (na + nb), "flops": 2 * count * _product(na, nb)}
    if op == "kara":  # two halvings from 8192 limbs, one from 4096
        levels = 2 if na >= 8192 else (1 if na >= 4096 else 0)
        return {"bytes": count * 32 * na, "flops": 2 * count * _product(na, na) * 0.75 ** levels}
    if op == "poly":  # four half products
        return {"bytes": count * 24 * na, "flops": 4 * count * _product(na, na)}
    nq = na - nb + 1
    return {"bytes": count * (8 * (na + nb + nq + nb) + 4), "flops": 2 * count * _division(na, nb)}


def tolerance(case):
    return "exact"


def _to_ints(t):
    return [int.from_bytes(row.tobytes(), "little") for row in t.cpu().numpy()]


def _to_limbs(values, n):
    raw = bytearray(b"".join(v.to_bytes(8 * n, "little") for v in values))
    return torch.frombuffer(raw, dtype=torch.int64).view(len(values), n).clone()


def exact(case, seed):
    """The same results from Python integers; None where they take long."""
    op, count = case["op"], case["count"]
    if op == "batch":
        return None
    na, nb = case["na"], case["nb"]
    if op in ("add", "sub", "chain"):
        cost = count * (2e-6 + 4e-9 * na)
    elif op == "divmod":
        cost = count * (1e-5 + 6e-9 * nb * (na - nb + 1))
    else:
        cost = count * (1e-5 + 2e-8 * (na * nb) ** 0.8) * (3 if op == "poly" else 1)
    if cost > 6:
        return None
    a, b = (_to_ints(t) for t in _operands(case, seed))
    mod = 1 << (64 * na)
    if op == "add":
        s = [x + y for x, y in zip(a, b)]
        return (_to_limbs([x % mod for x in s], na),
                torch.tensor([int(x >= mod) for x in s], dtype=torch.uint8))
    if op == "sub":
        return (_to_limbs([(x - y) % mod for x, y in zip(a, b)], na),
                torch.tensor([int(x < y) for x, y in zip(a, b)], dtype=torch.uint8))
    if op == "chain":
        s = [x + case["k"] * y for x, y in zip(a, b)]
        return (_to_limbs([x % mod for x in s], na),
                torch.tensor([x // mod for x in s], dtype=torch.uint8))
    if op in ("mul", "kara"):
        return _to_limbs([x * y for x, y in zip(a, b)], na + nb)
    if op == "poly":
        return _to_limbs([((x * x + y) * (y * y + y) + x * y) % mod for x, y in zip(a, b)], na)
    qr = [divmod(x, y) for x, y in zip(a, b)]
    return (_to_limbs([q for q, _ in qr], na - nb + 1), _to_limbs([r for _, r in qr], nb),
            torch.zeros(count, dtype=torch.int32))

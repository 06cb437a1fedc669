"""Performance cases of the library: what a program that multiplies under ABFT protection
has it do, through the public entry points of paper_0806_3121_gb300.abft.

A `step` is the whole protected product: encode the operands, multiply, verify (detect,
locate, correct) and, where a block was lost, rebuild it.  A `product` is encode and multiply
alone, for callers that keep the checksums.  A `chain` is two stacked products, the second one
taking the first one's checksums instead of encoding again.  A `group` is many independent
problems of uneven shapes in one launch.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_0806_3121_gb300 import abft


def listed():
    return [
        # The smallest problem in use: one 512^3 binary64 product whose single verify block
        # holds the whole result, one bit of the result flipped in memory before the verify.
        dict(name="f64_step_512", kind="step", dtype="f64", m=512, n=512, k=512, vb_r=512,
             vb_c=512, p=0, q=0, f=0, flips=1, erase=0, reread=1, dist="uniform"),
        # A binary64 problem whose sizes fit no tile, as applications bring them.
        dict(name="f64_step_ragged", kind="step", dtype="f64", m=1000, n=1501, k=777, vb_r=128,
             vb_c=100, p=0, q=0, f=0, flips=0, erase=0, reread=1, dist="normal"),
        # The block-grid workload (an 8 x 8 grid of 512-blocks): one block lost, three flips
        # in other blocks; verify, correct, rebuild.
        dict(name="f64_step_4096_grid8", kind="step", dtype="f64", m=4096, n=4096, k=4096,
             vb_r=512, vb_c=512, p=8, q=8, f=1, flips=3, erase=1, reread=1, dist="normal"),
        # Two stacked binary64 products that carry the checksums from one to the next.
        dict(name="f64_chain_2048", kind="chain", dtype="f64", m=2048, n=2048, k=2048, vb_r=256,
             vb_c=256, p=0, q=0, f=0, flips=0, erase=0, reread=1, dist="normal"),
        # A large binary64 product on a block grid, checksums kept for the caller.
        dict(name="f64_product_8192", kind="product", dtype="f64", m=8192, n=8192, k=8192,
             vb_r=512, vb_c=512, p=16, q=16, f=1, flips=0, erase=0, reread=1, dist="normal"),
        # The smallest tensor-core problem: launches and the host path count.
        dict(name="bf16_step_512", kind="step", dtype="bf16", m=512, n=512, k=512, vb_r=128,
             vb_c=256, p=0, q=0, f=0, flips=1, erase=0, reread=0, dist="normal"),
        # Ragged bf16 sizes, with the verify that reads the stored result back (the default).
        dict(name="bf16_step_ragged", kind="step", dtype="bf16", m=3001, n=2999, k=1111,
             vb_r=128, vb_c=256, p=0, q=0, f=0, flips=0, erase=0, reread=1, dist="normal"),
        # The large bf16 workload with three faults in the accumulators' outputs.
        dict(name="bf16_step_16384", kind="step", dtype="bf16", m=16384, n=16384, k=16384,
             vb_r=256, vb_c=256, p=0, q=0, f=0, flips=3, erase=0, reread=0, dist="normal"),
        # binary32 operands split in two bf16 pieces.
        dict(name="bf16x3_step_8192", kind="step", dtype="bf16x3", m=8192, n=8192, k=8192,
             vb_r=256, vb_c=256, p=0, q=0, f=0, flips=3, erase=0, reread=0, dist="normal"),
        # binary32 operands at binary32-level accuracy (three bf16 pieces).
        dict(name="bf16x6_step_16384", kind="step", dtype="bf16x6", m=16384, n=16384, k=16384,
             vb_r=256, vb_c=256, p=0, q=0, f=0, flips=3, erase=0, reread=0, dist="normal"),
        # e4m3 operands with one power-of-two scale per 128 x 128 block, rows of very
        # different magnitude.
        dict(name="fp8_step_16384", kind="step", dtype="fp8", m=16384, n=16384, k=16384,
             vb_r=256, vb_c=256, p=0, q=0, f=0, flips=5, erase=0, reread=0, dist="rows"),
        # Many independent bf16 problems, sizes uniform over multiples of 64 in [64, 2048],
        # one accumulator flip in 1 % of them: encode, the captured step, the report.
        dict(name="group_512", kind="group", dtype="bf16", count=512, lo=64, hi=2048,
             shape_seed=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["f64", "f64", "f64_grid", "chain", "bf16", "bf16", "bf16x3", "bf16x6",
                       "fp8", "group"])
    if kind == "group":
        return dict(kind="group", dtype="bf16", count=_log_int(rng, 16, 640), lo=64,
                    hi=rng.choice([512, 1024, 2048]), shape_seed=rng.randrange(1 << 20))
    if kind == "f64_grid":
        p = rng.randint(2, 8)
        bs = _log_int(rng, 64, 512)
        f = rng.choice([1, 1, 2])
        return dict(kind="step", dtype="f64", m=p * bs, n=p * bs, k=_log_int(rng, 256, 4096),
                    vb_r=bs, vb_c=bs, p=p, q=p, f=f, flips=rng.randint(0, 2), erase=1, reread=1,
                    dist="normal")
    hi = {"f64": 4096, "chain": 2500}.get(kind, 12000)
    m, n, k = (_log_int(rng, 256, hi) for _ in range(3))
    if rng.random() < 0.3:
        m, n, k = (max(256, v // 128 * 128) for v in (m, n, k))
    dtype = "f64" if kind in ("f64", "chain") else kind
    vb_r = rng.choice([128, 256])
    vb_c = rng.choice([128, 256])
    if dtype == "f64" and rng.random() < 0.5:
        vb_r, vb_c = rng.randint(32, 256), rng.randint(32, 256)
    return dict(kind="chain" if kind == "chain" else "step", dtype=dtype, m=m, n=n, k=k,
                vb_r=vb_r, vb_c=vb_c, p=0, q=0, f=0,
                flips=0 if kind == "chain" else rng.randint(0, 3), erase=0,
                reread=1 if dtype == "f64" else rng.randint(0, 1),
                dist="rows" if dtype == "fp8" else
                rng.choice(["normal", "uniform", "rows"] if dtype == "f64" else
                           ["normal", "uniform"]))


# ------------------------------------------------------------------ inputs

def _ceil(x, q):
    return -(-x // q) * q


def _values(rows, cols, dist, dtype, g):
    if dist == "normal":
        return torch.randn(rows, cols, generator=g, device="cuda", dtype=dtype)
    x = torch.rand(rows, cols, generator=g, device="cuda", dtype=dtype).mul_(2).sub_(1)
    if dist == "rows":  # one magnitude in [1e-2, 1e2] per row
        x *= 10.0 ** (torch.rand(rows, 1, generator=g, device="cuda", dtype=dtype) * 4 - 2)
    return x


def _padded(x, q):
    """x in rows whose length is a multiple of q elements."""
    r, c = x.shape
    if c % q == 0:
        return x.contiguous()
    out = torch.zeros(r, _ceil(c, q), dtype=x.dtype, device=x.device)
    out[:, :c] = x
    return out


def _quantised(x):
    """(e4m3 codes, binary32 power-of-two scale per 128 x 128 block)."""
    r, c = x.shape
    br, bc = -(-r // 128), -(-c // 128)
    full = torch.zeros(br * 128, bc * 128, device=x.device)
    full[:r, :c] = x
    t = full.view(br, 128, bc, 128)
    amax = t.abs().amax(dim=(1, 3))
    s = torch.exp2(torch.ceil(torch.log2(torch.where(amax > 0, amax, 448.0) / 448.0)))
    codes = (t / s[:, None, :, None]).to(torch.float8_e4m3fn).view(br * 128, bc * 128)[:r, :c]
    return codes.contiguous().view(torch.uint8), s.float().contiguous()


def _operands(case, seed):
    """A and B as the caller holds them (rows padded where the dtype asks for aligned rows),
    and their block scales."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    m, n, k, dt = case["m"], case["n"], case["k"], case["dtype"]
    fp = torch.float64 if dt == "f64" else torch.float32
    A, B = (_values(r, c, case["dist"], fp, g) for r, c in ((m, k), (k, n)))
    if dt == "bf16":
        return _padded(A.to(torch.bfloat16), 8), _padded(B.to(torch.bfloat16), 8), None, None
    if dt == "fp8":
        (qa, sa), (qb, sb) = _quantised(A), _quantised(B)
        return _padded(qa, 16), _padded(qb, 16), sa, sb
    return A, B, None, None


def _raising_bit(x, f64):
    """The exponent bit whose flip makes a result of value x larger by 2^64 (2^512) or more:
    a fault that no rounding hides."""
    return (61 if f64 else 29) if abs(x) >= 2 else (62 if f64 else 30)


def _faults(case, seed, A, B, sa, sb):
    """(row, column, bit) flips in distinct verify blocks and the lost block, if any."""
    r = random.Random(seed)
    m, n = case["m"], case["n"]
    lost = [(r.randrange(case["p"]), r.randrange(case["q"]))] if case["erase"] else []
    bs, bc = (m // case["p"], n // case["q"]) if case["p"] else (1, 1)
    used, flips = set(), []
    for t in range(200):
        if len(flips) == case["flips"]:
            break
        i, j = r.randrange(m), r.randrange(n)
        if (i // bs, j // bc) in lost:
            continue
        lines = {("r", i // case["vb_r"]), ("c", j // case["vb_c"])}
        if lines & used and (m > case["vb_r"] and n > case["vb_c"]):
            continue
        if flips and not (m > case["vb_r"] and n > case["vb_c"]):
            break
        used |= lines
        a = _f64(case, A[i:i + 1], None if sa is None else sa[i // 128:i // 128 + 1], 1, case["k"])
        b = _f64(case, B[:, j:j + 1], None if sb is None else sb[:, j // 128:j // 128 + 1],
                 case["k"], 1)
        flips.append((i, j, _raising_bit(float(a @ b), case["dtype"] == "f64")))
    return flips, lost


class _Group:
    """Problems of one group in three flat buffers, the bound handle and its captured step."""

    def __init__(self, case, seed):
        r = random.Random(case["shape_seed"])
        lo, hi = case["lo"] // 64, case["hi"] // 64
        self.shapes = [tuple(64 * r.randint(lo, hi) for _ in range(3))
                       for _ in range(case["count"])]
        g = torch.Generator(device="cuda").manual_seed(seed)
        na, nb, nc = (sum(x * y for x, y in v) for v in zip(
            *(((m, k), (k, n), (m, n)) for m, n, k in self.shapes)))
        self.A = torch.randn(na, generator=g, device="cuda").to(torch.bfloat16)
        self.B = torch.randn(nb, generator=g, device="cuda").to(torch.bfloat16)
        self.C = torch.zeros(nc, device="cuda")
        probs, self.at, oa, ob, oc = [], [], 0, 0, 0
        for m, n, k in self.shapes:
            self.at.append((oa, ob, oc))
            probs.append((m, n, k, self.A[oa:].data_ptr(), self.B[ob:].data_ptr(),
                          self.C[oc:].data_ptr()))
            oa, ob, oc = oa + m * k, ob + k * n, oc + m * n
        self.g = abft.abft_group_create(probs)
        self.ws = torch.zeros(abft.abft_group_workspace_bytes(self.g), dtype=torch.uint8,
                              device="cuda")
        self.stream = torch.cuda.Stream()
        self.stream.wait_stream(torch.cuda.current_stream())
        abft.abft_group_bind(self.g, self.ws, self.stream)
        rf = random.Random(seed + 1)
        flips = []
        for q in sorted(rf.sample(range(case["count"]), max(1, case["count"] // 100))):
            (m, n, k), (oa, ob, _) = self.shapes[q], self.at[q]
            i, j = rf.randrange(m), rf.randrange(n)
            x = self.A[oa + i * k:oa + (i + 1) * k].double() @ self.B[ob + j:ob + k * n:n].double()
            flips.append((q, i, j, _raising_bit(float(x), False)))
        abft.abft_group_set_epilogue_faults(self.g, flips, self.stream)
        abft.abft_group_capture(self.g, True, self.stream)

    def __del__(self):
        if getattr(self, "g", None):
            abft.abft_group_destroy(self.g)


def prepare(case, seed):
    if case["kind"] == "group":
        return case, _Group(case, seed)
    m, n, k, dt = case["m"], case["n"], case["k"], case["dtype"]
    A, B, sa, sb = _operands(case, seed)
    vb_r, vb_c = min(case["vb_r"], m), min(case["vb_c"], n)
    desc = abft.make_desc(m, n, k, dt, vb_r, vb_c, case["p"], case["q"], lda=A.shape[1],
                          ldb=B.shape[1], grid_f=case["f"])
    out = torch.float64 if dt == "f64" else torch.float32
    S = dict(A=A, B=B, sa=sa, sb=sb, desc=desc,
             C=torch.zeros(m, n, dtype=out, device="cuda"),
             ws=torch.zeros(abft.abft_workspace_bytes(desc), dtype=torch.uint8, device="cuda"))
    S["flips"], S["lost"] = _faults(case, seed, A, B, sa, sb)
    if dt != "f64" and S["flips"]:  # compute faults, armed on the workspace
        abft.abft_set_epilogue_faults(desc, S["ws"], S["flips"])
    if case["kind"] == "product":
        L = abft.abft_workspace_layout(desc)
        S["E"] = S["ws"][L.E:L.E + 8 * L.R * n].view(torch.float64).view(L.R, n)
        S["F"] = S["ws"][L.F:L.F + 8 * L.Cc * m].view(torch.float64).view(m, L.Cc)
    if case["kind"] == "chain":  # D: n x k, so the second result is m x k
        g = torch.Generator(device="cuda").manual_seed(seed + 7919)
        S["D"] = _values(n, k, case["dist"], torch.float64, g)
        S["desc2"] = abft.make_desc(m, k, n, dt, vb_r, min(case["vb_c"], k))
        S["C2"] = torch.zeros(m, k, dtype=out, device="cuda")
        S["ws2"] = torch.zeros(abft.abft_workspace_bytes(S["desc2"]), dtype=torch.uint8,
                               device="cuda")
    return case, S


def _report(faults):
    return np.array([[f["problem"], f["row"], f["col"], f["kind"]] for f in faults],
                    dtype=np.int64).reshape(-1, 4)


def run(state):
    case, S = state
    if case["kind"] == "group":
        S.stream.wait_stream(torch.cuda.current_stream())
        abft.abft_group_encode(S.g, S.stream)
        abft.abft_group_launch(S.g, S.stream)
        status, faults, count = abft.abft_group_report(S.g, stream=S.stream)
        return {"C": S.C, "status": status, "count": count, "faults": _report(faults)}
    d, C, ws = S["desc"], S["C"], S["ws"]
    abft.abft_encode(d, S["A"], S["B"], ws, S["sa"], S["sb"])
    abft.abft_gemm(d, S["A"], S["B"], C, ws, S["sa"], S["sb"])
    if case["kind"] == "product":
        return {"C": C, "E": S["E"], "F": S["F"]}
    if case["dtype"] == "f64" and S["flips"]:  # memory faults in the stored result
        abft.abft_inject_bitflips(d, C, S["flips"])
    for bi, bj in S["lost"]:
        abft.abft_erase_block(d, C, bi, bj)
    status, faults, count = abft.abft_verify_correct(d, C, ws, erased=S["lost"],
                                                     reread_C=case["reread"])
    out = {"C": C, "status": status, "count": count, "faults": _report(faults)}
    for bi, bj in S["lost"]:
        out["rebuilt"] = abft.abft_recover_block(d, C, ws, bi, bj)[0]
    if case["kind"] == "chain":
        d2 = S["desc2"]
        abft.abft_encode_chained(d2, C, S["D"], S["ws2"], left=(d, ws))
        abft.abft_gemm(d2, C, S["D"], S["C2"], S["ws2"])
        out["status2"], _, out["count2"] = abft.abft_verify_correct(d2, S["C2"], S["ws2"],
                                                                    reread_C=1)
        out["C2"] = S["C2"]
    return out


def work(case):
    """Operands read once, results written once; the products of the data and of the
    unweighted and weighted checksums of every verify block (and the block checksums)."""
    if case["kind"] == "group":
        r = random.Random(case["shape_seed"])
        lo, hi = case["lo"] // 64, case["hi"] // 64
        b = fl = 0
        for _ in range(case["count"]):
            m, n, k = (64 * r.randint(lo, hi) for _ in range(3))
            b += 2 * k * (m + n) + 4 * m * n
            fl += 2 * k * (m * n + 2 * -(-m // 128) * n + 2 * m * -(-n // 256))
        return {"bytes": b, "flops": fl}
    m, n, k = case["m"], case["n"], case["k"]
    ein, eout = {"f64": (8, 8), "bf16": (2, 4), "fp8": (1, 4)}.get(case["dtype"], (4, 4))

    def product(m, n, k):
        rows = 2 * -(-m // case["vb_r"]) + (case["f"] * (m // case["p"]) if case["p"] else 0)
        cols = 2 * -(-n // case["vb_c"])
        return ein * k * (m + n) + eout * m * n, 2 * k * (m * n + rows * n + m * cols)

    b, fl = product(m, n, k)
    if case["kind"] == "chain":
        b2, fl2 = product(m, k, n)
        b, fl = b + b2, fl + fl2
    return {"bytes": b, "flops": fl}


def _f64(case, x, s, rows, cols):
    """An operand's values in binary64."""
    if case["dtype"] != "fp8":
        return x[:, :cols].double()
    v = x[:, :cols].view(torch.float8_e4m3fn).double()
    s = s.double().repeat_interleave(128, 0)[:rows].repeat_interleave(128, 1)[:, :cols]
    return v * s


def exact(case, seed):
    if case["kind"] == "group":
        G = _Group(case, seed)
        C = torch.empty(G.C.numel(), dtype=torch.float64, device="cuda")
        for (m, n, k), (oa, ob, oc) in zip(G.shapes, G.at):
            torch.mm(G.A[oa:oa + m * k].view(m, k).double(),
                     G.B[ob:ob + k * n].view(k, n).double(), out=C[oc:oc + m * n].view(m, n))
        return {"C": C, "status": None, "count": None, "faults": None}
    m, n, k = case["m"], case["n"], case["k"]
    A, B, sa, sb = _operands(case, seed)
    A, B = _f64(case, A, sa, m, k), _f64(case, B, sb, k, n)
    out = {"C": A @ B}
    if case["kind"] == "product":
        bs = m // case["p"]

        def sums(x, vb):  # (plain sum, sum weighted by (t + 1) / 2^ceil(log2 vb)) per block
            w = torch.arange(1, vb + 1, device="cuda", dtype=torch.float64)
            w = w / 2.0 ** math.ceil(math.log2(vb))
            rows = []
            for t in range(0, x.shape[0], vb):
                c = x[t:t + vb]
                rows += [c.sum(0), w[:c.shape[0]] @ c]
            return torch.stack(rows)

        S = A.view(case["p"], bs, k).sum(0)
        out["E"] = torch.cat([sums(A, case["vb_r"]) @ B, S @ B])
        out["F"] = A @ sums(B.t().contiguous(), case["vb_c"]).t()
    else:
        out.update(status=None, count=None, faults=None)
    if case["erase"]:
        out["rebuilt"] = None
    if case["kind"] == "chain":
        g = torch.Generator(device="cuda").manual_seed(seed + 7919)
        out.update(status2=None, count2=None,
                   C2=out["C"] @ _values(n, k, case["dist"], torch.float64, g))
    return out

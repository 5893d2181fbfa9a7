"""Performance cases of the ORBGRAND decoder: the calls its users make.

Each case is one call of a public entry point of
``paper_2202_13951_gb300.orbg`` on BPSK/AWGN blocks (the channel of
``workloads.awgn_llr``, drawn on the device), with the codes, Eb/N0 ranges and
query caps of the repository's own benchmark and tests.  Outputs are whole
numbers throughout: codeword bytes, query counts, flags, model records.
"""
import functools
import math

import numpy as np
import torch

from paper_2202_13951_gb300 import orbg, workloads

#: name -> (codes, Eb/N0 range in dB, mean queries a block there at the caps
#: below).  More than one code: equal shares of them, in random order.
SETS = {
    "rlc64": (lambda: [workloads.config1_code()], (5.0, 5.0), 17),
    "bch127": (lambda: [workloads.config2_code()], (4.0, 7.0), 300),
    "capolar128": (lambda: [workloads.config3_code()], (3.0, 6.0), 119_000),
    "capolar256": (lambda: [workloads.capolar256_code()], (5.0, 5.3), 4_100),
    "rlc4": (workloads.config4_codes, (4.0, 7.0), 7_100),
    "serve3": (workloads.config5_codes, (3.0, 7.0), 33_000),
    "paper256": (workloads.paper256_codes, (4.0, 7.0), 46_000),
}
#: the one-line and three-segment orders fitted to bch127's mean ordered |LLR|
LINE = (5, 1)
MODEL = ((7, 17), (3, 37, 58), (5, 2, 1))


@functools.lru_cache(maxsize=None)
def _codes(name, n, r):
    """The codes of a set; "rlc": one random linear code of length n with r
    parity bits."""
    if name == "rlc":
        return [workloads.rlc(n, n - r, seed=7)]
    return SETS[name][0]()


def _case(name, form, codes, blocks, cap, n=0, r=0, lines=0, divisible=False):
    c = {"form": form, "codes": codes, "blocks": blocks, "cap": cap, "n": n, "r": r,
         "lines": lines, "divisible": divisible}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a receiver that decodes one slot's few blocks as they come in: the
        # smallest call, all latency
        _case("plain_rlc64_32", "plain", "rlc64", 32, 100_000),
        # a ragged small batch of one code
        _case("batched_bch127_257", "batched", "bch127", 257, 1_000_000),
        # one admitted batch of the serving loop: its three codes mixed
        _case("mixed_serve3_8191", "mixed", "serve3", 8_191, 1_000_000),
        # the single-launch form on an ordinary batch
        _case("plain_bch127_100k", "plain", "bch127", 100_000, 1_000_000),
        # a large batch of one short-search code: per-block work counts
        _case("batched_bch127_400k", "batched", "bch127", 400_000, 1_000_000),
        # long searches, two-word syndromes: per-query work counts
        _case("batched_capolar128_100k", "batched", "capolar128", 100_000, 1_000_000),
        # the headline: four codes of very uneven search depth in one call
        _case("mixed_rlc4_1m", "mixed", "rlc4", 1_000_000, 1_000_000),
        # the [256, 234] family at the paper's deep cap, an odd block count
        _case("mixed_paper256_100k", "mixed", "paper256", 100_003, 5_000_000),
        # full ORBGRAND with one three-segment model for the code
        _case("model_bch127_100k", "model", "bch127", 100_000, 1_000_000),
        # full ORBGRAND with three lines fitted to every block
        _case("fitted3_bch127_100k", "fitted", "bch127", 100_000, 1_000_000, lines=3),
        # the same at the paper's operating point, a few very long searches
        _case("fitted3_capolar256_20k", "fitted", "capolar256", 20_000, 5_000_000, lines=3),
        # a program with its data in pinned host memory
        _case("host_rlc4_262k", "host", "rlc4", 262_144, 1_000_000),
    ]


def _log(rng, lo, hi):
    """A whole number of lo..hi, uniform in its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    form = rng.choice(["plain", "batched", "batched", "mixed", "mixed", "line", "model",
                       "fitted", "fitted1", "host"])
    if form in ("plain", "batched"):
        codes = rng.choice(["rlc64", "bch127", "capolar128", "rlc", "rlc"])
        if codes == "capolar128":
            return _case(None, form, codes, _log(rng, 1, 100_000 if form == "batched" else 2_000),
                         _log(rng, 10_000, 1_000_000))
        n = r = 0
        if codes == "rlc":
            # random linear codes of any length, odd ones among them
            n = _log(rng, 40, 256)
            r = rng.randint(8, min(24, n // 4))
        most = 400_000 if codes in ("rlc64", "bch127") and form == "batched" else 60_000
        return _case(None, form, codes, _log(rng, 1, most), _log(rng, 1_000, 1_000_000), n, r)
    if form in ("mixed", "host"):
        codes = rng.choice(["rlc4", "rlc4", "serve3", "paper256"])
        most = 1_000_000 if codes == "rlc4" and form == "mixed" else 262_144
        if codes != "rlc4":
            most = 50_000
        return _case(None, form, codes, _log(rng, 1, most), _log(rng, 10_000, 1_000_000))
    if form == "fitted":
        codes = rng.choice(["rlc64", "bch127", "capolar256"])
        return _case(None, form, codes, _log(rng, 1, 10_000 if codes == "capolar256" else 80_000),
                     _log(rng, 10_000, 1_000_000), lines=rng.randint(1, 4),
                     divisible=rng.random() < 0.5)
    if form == "fitted1":
        return _case(None, form, rng.choice(["rlc64", "bch127"]), _log(rng, 1, 60_000),
                     _log(rng, 10_000, 100_000), lines=1)
    return _case(None, form, "bch127", _log(rng, 1, 300_000), _log(rng, 10_000, 1_000_000))


def _range(case):
    return SETS[case["codes"]][1] if case["codes"] in SETS else (4.5, 7.0)


def _blocks(code, ebn0, gen):
    """One BPSK/AWGN block of `code` per entry of ebn0 (dB): LLRs [B][n]."""
    dev = ebn0.device
    B = ebn0.numel()
    info = torch.randint(0, 2, (B, code.k), generator=gen, device=dev).float()
    c = (info @ torch.from_numpy(code.G).to(dev).float()) % 2.0
    s2 = 1.0 / (2.0 * (code.k / code.n) * torch.pow(10.0, ebn0 / 10.0))[:, None]
    y = (2.0 * c - 1.0) + torch.sqrt(s2) * torch.randn((B, code.n), generator=gen, device=dev)
    return (2.0 * y / s2).contiguous()


class State:
    """The handles a program keeps, one call's inputs and, for the host
    form, its output buffers."""


def prepare(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    form, B, cap = case["form"], case["blocks"], case["cap"]
    codes = _codes(case["codes"], case["n"], case["r"])
    lo, hi = _range(case)
    ebn0 = lo + (hi - lo) * torch.rand(B, generator=gen, device=dev)
    s = State()
    s.form, s.cap, s.lines, s.divisible = form, cap, case["lines"], case["divisible"]
    order = {"line": LINE} if form == "line" else {"model": MODEL} if form == "model" else {}
    # decode_fitted does not use the handle's query-order tables
    depth = 1_000 if form == "fitted" else cap
    s.codes = [orbg.Code(c.H, n=c.n, k=c.k, max_query_cap=depth, **order) for c in codes]
    if form in ("batched", "line", "model", "mixed", "host"):
        s.set = orbg.CodeSet(s.codes)
    if form == "fitted1":
        s.fitted = orbg.Fitted(s.codes[0])
    if form not in ("mixed", "host"):
        s.llr = _blocks(codes[0], ebn0, gen)
        return s
    # equal shares of the codes, in random order
    cid = (torch.arange(B, device=dev) % len(codes))[torch.randperm(B, generator=gen, device=dev)]
    ns = torch.tensor([c.n for c in codes], device=dev)[cid]
    off = torch.cumsum(ns, 0) - ns
    s.total = int(ns.sum())
    s.llr = torch.empty(s.total, dtype=torch.float32, device=dev)
    for j, c in enumerate(codes):
        at = torch.nonzero(cid == j).flatten()
        s.llr[off[at][:, None] + torch.arange(c.n, device=dev)] = _blocks(c, ebn0[at], gen)
    s.code_id, s.off = cid.to(torch.int32), off
    if form == "host":
        def pinned(t):
            h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
            return h.copy_(t)
        s.code_id, s.off, s.llr = pinned(s.code_id), pinned(s.off), pinned(s.llr)
        s.out = (torch.zeros(s.total, dtype=torch.uint8, pin_memory=True),
                 torch.zeros(B, dtype=torch.int32, pin_memory=True),
                 torch.zeros(B, dtype=torch.uint8, pin_memory=True))
    return s


def run(s):
    if s.form == "plain":
        return orbg.decode(s.codes[0], s.llr, s.cap)
    if s.form == "fitted":
        return orbg.decode_fitted(s.codes[0], s.llr, s.cap, s.lines, s.divisible)
    if s.form == "fitted1":
        return s.fitted.decode(s.llr, s.cap)
    if s.form == "mixed":
        return orbg.decode_batched(s.set, s.llr, s.cap, code_id=s.code_id, llr_offset=s.off,
                                   cw_offset=s.off, n_total=s.total)
    if s.form == "host":
        cw, q, ab = s.out
        orbg.orbg_decode_batched(s.set.handle, s.code_id, s.off, s.llr, s.off.numel(),
                                 s.cap, cw, s.off, q, ab, torch.cuda.current_stream())
        return s.out
    return orbg.decode_batched(s.set, s.llr, s.cap)


def work(case):
    """Bytes: LLRs in, codeword, query count and flag out (and a mixed call's
    code ids and offsets in, a fitted call's model record out).  flops: 32-bit
    integer operations, n log2 n compares of a block's sort and two for each
    of its queries (one XOR, one compare) at the set's mean query count."""
    codes = _codes(case["codes"], case["n"], case["r"])
    n = float(np.mean([c.n for c in codes]))
    per = 5.0 * n + 5.0
    if case["form"] in ("mixed", "host"):
        per += 4 + 8  # one offset array serves LLRs and codewords
    if case["form"] in ("fitted", "fitted1"):
        per += 4 * orbg.ORBG_FIT_STRIDE
    queries = SETS[case["codes"]][2] if case["codes"] in SETS else 2.0 ** case["r"] / 500.0
    ops = n * math.ceil(math.log2(n)) + 2.0 * min(case["cap"], queries)
    return {"bytes": case["blocks"] * per, "flops": case["blocks"] * ops}


def exact(case, seed):
    """Every output is a whole number, equal or wrong: no 64-bit value."""
    return None

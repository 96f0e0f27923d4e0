"""Time estimate of a contraction call from the library's compiled launch list.

The plan compiler decides, for every pairwise step, the kernel family, the
operand layouts (and so the permutes) and which operands a launch shares
between its items; qx_describe_plan lists the steps.  This prices each
launch on one GB300: its bytes (operands read once per item, an
operand of a lower dependence level once per launch, the result written
once) at the HBM rate its kernel family reaches, or its complex flops
(8 M K N) at the family's arithmetic rate, whichever takes longer, plus a
launch cost, and sums the launches.  Steps that run as one launch are priced
once: a call's prologue (all steps with a chain= number), and a segment (the
steps of a seg= number) where the library runs it so, by the library's own
rule.  The rates were measured per family on the 36-qubit sliced workload.  Against
calls on one stream, as a serving lane makes them (31 calls of 33 us to 74 ms:
the benchmark's and seven serving plans, 1 to 1024 bitstrings), the sums lie at
0.81 to 1.39 of the measured times.  With concurrent streams the calls whose
launches are short take down to 0.5 of the estimate.
The server uses the estimate for admission, planners to rank plans.
"""
from __future__ import annotations

# kernel family -> (complex flop/s, or None for data movement; bytes/s).  "tc_direct_kb": the direct
# tensor-core kernel with B' resident per CTA (B shared by every item, one tile wide)
GB300_LAUNCH_RATES = {"permute": (None, 6.0e12), "gather": (26e12, 4.7e12), "tc_direct": (150e12, 3.5e12),
                      "tc_direct_kb": (150e12, 4.8e12), "tc_prep": (260e12, 5.0e12), "gemm": (35e12, 4.0e12),
                      "dot_perm": (35e12, 5.0e12)}
_LEVEL = {"shared": 0, "slice": 1, "pair": 2}
_SM, _CLOCK, _WARPS = 152, 1.9e9, 4  # SMs, their clock, warps that an SM issues from at a time
_TILE16 = 64e9  # complex flop/s of the GEMM on one SM, on the 16 x 16 tiles of a product with few outputs
_SHORT = 16e12  # complex flop/s of the GEMM with a short side of at most 4
_BANKS = 3.5  # issue time of a segment against its listed clocks (shared-memory bank conflicts)


def _regions(field):
    out = []
    for part in field.split(",") if field else ():
        reg, rest = part.split(":")
        out.append((reg, int(rest.split("+")[1])))
    return out


def _step_time(kind, level, kv, items, rates):
    """Seconds of one step as a launch of its own, without the launch cost."""
    it = items[_LEVEL[level]]
    nbytes = sum(8.0 * e * (it if r == level else items[_LEVEL[r]]) for r, e in _regions(kv.get("reads", "")))
    nbytes += sum(8.0 * e * it for r, e in _regions(kv.get("writes", "")))
    if kind == "tc_direct" and "m" in kv:
        # the launch picks the resident-B' variant when B is shared by every item, one 128- or 64-wide
        # tile (N = 64 or 32) and at most 4 or 8 K stages of 32 reals, and A is not kept per slice
        regs = _regions(kv.get("reads", ""))
        n, k = int(kv["n"]), int(kv["k"])
        if len(regs) == 2 and regs[1][0] == "shared" and regs[0][0] == level and (
                (n == 6 and (2 << k) // 32 <= 4) or (n == 5 and (2 << k) // 32 <= 8)):
            kind = "tc_direct_kb"
    fr, br = rates.get(kind, (35e12, 4.0e12))
    t = nbytes / br
    if fr and "m" in kv:
        m, k, n = int(kv["m"]), int(kv["k"]), int(kv["n"])
        if kind == "gemm" and min(m, n) <= 2:
            fr = min(fr, _SHORT)
        t = max(t, 8.0 * 2.0 ** (m + k + n) * it / fr)
        # few tiles: one tile's sum over K on its SM (128 x 64 on the tensor cores; the GEMM takes tiles of
        # 16 x 16 then)
        if kind.startswith("tc_"):
            t = max(t, 8.0 * 2.0 ** (7 + k + 6) * _SM / fr)
        elif kind == "gemm":
            t = max(t, 8.0 * 2.0 ** (min(m, 4) + k + min(n, 4)) / _TILE16)
    return t


def _segment_time(kv, n_items, sms=_SM):
    """Seconds of a segment's launch over n_items items on `sms` SMs: its stages one after another, or
    its issue time."""
    return max(4e-6 + 0.35e-6 * int(kv["stages"]),
               _BANKS * n_items * float(kv["clocks"]) / (sms * _WARPS) / _CLOCK)


def parse(desc):
    """The steps of a qx_describe_plan listing: (kernel family, dependence level, fields)."""
    rows = (line.split() for line in desc.splitlines())
    return [(f[2], f[3], dict(x.split("=", 1) for x in f[4:] if "=" in x)) for f in rows]


def launches(desc, items, rates=GB300_LAUNCH_RATES, launch=4e-6):
    """(dependence level, seconds) of every launch of a batch from a qx_describe_plan listing (or its
    parsed steps); items: the launches' items by level (1, slices, (slice, bitstring) pairs)."""
    out, chains, segs = [], [], {}
    for kind, name, kv in parse(desc) if isinstance(desc, str) else desc:
        level = _LEVEL[name]
        if "chain" in kv:  # all chains run in one launch, a CTA each
            if "stages" in kv:
                chains.append(_segment_time(kv, 1, 1))
            continue
        t = _step_time(kind, name, kv, items, rates) + launch
        if "seg" not in kv:
            out.append((level, t))
            continue
        steps = segs.setdefault(kv["seg"], [])
        steps.append((level, t))
        if "stages" in kv:  # the segment's last step
            # the library's rule (seg_pays): one launch against one per step, 2.5 us or its bytes each
            one = _segment_time(kv, items[level])
            apart = max(2.5e-6 * len(steps), items[level] * float(kv["step_bytes"]) / 4.5e12)
            out += [(level, one)] if one < apart else steps
    if chains:
        out.insert(0, (0, max(max(chains), sum(chains) / _SM)))
    return out


def launch_list_time(desc, n_slices, n_bits, rates=GB300_LAUNCH_RATES, launch=4e-6, max_items=None, kept=False):
    """Seconds of one call over n_slices slices and n_bits bitstrings from a qx_describe_plan listing (or
    its parsed steps; launches priced one after another), with the launches that every call has: two
    clears, the sums over the slices (0.3 us each, in order) and their end.  max_items: (slice, bitstring)
    pairs that a batch of the workspace holds, at least n_bits of them; None: all.  kept: the invariant
    intermediates are kept from an earlier call (qx_set_memo)."""
    per = n_slices if max_items is None else max(1, min(n_slices, max_items // n_bits))
    batches = -(-n_slices // per)
    listed = launches(desc, (1, per, per * n_bits), rates, launch)
    once, per_batch = (sum(t for level, t in listed if (level > 0) == later) for later in (False, True))
    return (0.0 if kept else once) + batches * (per_batch + launch) + 3 * launch + 0.3e-6 * n_slices

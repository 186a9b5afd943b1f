"""What a user has this library do, as timed cases: settings for a permutation, and a payload through them.

A case names the way in (the public calls a program makes), the sizes, the element type of the payload and the
kind of permutation:

  way      "calls"   binding.route, then binding.apply on the settings (the usage of the README)
           "apply"   binding.apply on settings that were computed once and are kept
           "padded"  benes_route_padded, then benes_apply_padded: rows whose length is no power of two
           "plan"    Plan.launch: the same route + apply on fixed buffers, replayed
           "host"    benes_route_apply_host: pinned host buffers in and out, settings wanted back
  n_elems  elements of a permutation (a power of two but for "padded")
  batch    independent permutations
  dtype    "i32", "f32" or "i64" payload elements
  perm     "random", "cycle" (one cycle through all elements), "shift", "transpose", "bitrev", "identity"
"""
import math

import torch

from paper_1912_04050_b200 import binding

DTYPES = {"i32": torch.int32, "f32": torch.float32, "i64": torch.int64}
BYTES = {"i32": 4, "f32": 4, "i64": 8}


def case(way, n_elems, batch, dtype, perm="random"):
    return {"way": way, "n_elems": n_elems, "batch": batch, "dtype": dtype, "perm": perm}


def listed():
    def named(name, *a):
        return dict(case(*a), name=name)

    return [
        # the smallest calls: a few short permutations (a sorter's or a crossbar's port map), where latency counts
        named("calls 32 x 2^6 f32", "calls", 1 << 6, 32, "f32"),
        # one permutation that one thread block finishes
        named("calls 2^10 i32", "calls", 1 << 10, 1, "i32"),
        # many short permutations, independent of one another: the batched configuration
        named("calls 16384 x 2^8 i32", "calls", 1 << 8, 16384, "i32"),
        # the same amount of data and more in medium rows, as when the rows of a matrix are shuffled
        named("calls 4096 x 2^12 f32", "calls", 1 << 12, 4096, "f32"),
        # rows one size above what a block's shared memory holds
        named("calls 256 x 2^16 i32", "calls", 1 << 16, 256, "i32"),
        # one permutation of a million elements, the low end of the headline's range
        named("calls 2^20 f32", "calls", 1 << 20, 1, "f32"),
        # a structured permutation: the index map of a 4096 x 4096 matrix transpose
        named("calls 2^24 i32 transpose", "calls", 1 << 24, 1, "i32", "transpose"),
        # the headline: the largest single permutation with a 64-bit payload
        named("calls 2^26 i64", "calls", 1 << 26, 1, "i64"),
        # rows whose length is no power of two
        named("padded 3 x 1000003 i64", "padded", 1000003, 3, "i64"),
        # one direction alone: fixed networks, new payloads every time
        named("apply 4 x 2^22 i64", "apply", 1 << 22, 4, "i64"),
        # a program that runs the same buffers again and again keeps a plan
        named("plan 2^18 f32", "plan", 1 << 18, 1, "f32"),
        # data that lives in host memory, both ways over the bus
        named("host 2^22 i64", "host", 1 << 22, 1, "i64"),
    ]


# log2 of the elements of all permutations together, per way in
RANGES = {"calls": (6.0, 25.5), "apply": (6.0, 25.5), "padded": (8.0, 23.0), "plan": (10.0, 22.0), "host": (12.0, 24.0)}


def draw(rng):
    """One more case: the ways in by how often they are used, sizes spread over the logarithm of their range."""
    way = rng.choice(["calls"] * 6 + ["apply"] * 2 + ["padded"] * 2 + ["plan"] + ["host"])
    lo, hi = RANGES[way]
    total = rng.uniform(lo, hi)
    dtype = rng.choice(["i32", "f32", "i64"])
    perm = rng.choice(["random"] * 5 + ["cycle", "shift", "transpose", "bitrev"])
    if way == "padded":
        row = total if rng.random() < 0.5 else rng.uniform(min(5.0, total), total)
        n_elems = max(3, int(2.0 ** row)) | 1                  # odd
        return case(way, n_elems, max(1, int(2.0 ** total) // n_elems), dtype)
    # one permutation in half of the cases, else a batch of any (mostly odd) count
    log2n = int(total) if rng.random() < 0.5 else rng.randint(5, int(total))
    return case(way, 1 << log2n, max(1, int(2.0 ** (total - log2n))), dtype, perm)


def permutations(c, gen):
    """(batch, n_elems) int32 permutations on the GPU."""
    N, B = c["n_elems"], c["batch"]
    kind = c["perm"]
    if kind == "random" and B <= 64:
        return torch.stack([torch.randperm(N, generator=gen, device="cuda").to(torch.int32) for _ in range(B)])
    if kind == "random":
        return torch.rand((B, N), generator=gen, device="cuda").argsort(dim=1, stable=True).to(torch.int32)
    j = torch.arange(N, device="cuda")
    log2n = N.bit_length() - 1
    if kind == "cycle":
        order = torch.randperm(N, generator=gen, device="cuda")
        p = torch.empty_like(order)
        p[order] = order.roll(-1)
    elif kind == "shift":
        p = (j + 1) % N
    elif kind == "transpose":
        rows = 1 << (log2n // 2)
        cols = N // rows
        p = (j % cols) * rows + j // cols
    elif kind == "bitrev":
        p = torch.zeros_like(j)
        for b in range(log2n):
            p |= ((j >> b) & 1) << (log2n - 1 - b)
    else:
        p = j
    return p.to(torch.int32).expand(B, N).contiguous()


def payload(c, gen):
    shape = (c["batch"], c["n_elems"])
    if c["dtype"] == "f32":
        return torch.rand(shape, generator=gen, device="cuda")
    top = 1 << (31 if c["dtype"] == "i32" else 62)
    return torch.randint(0, top, shape, generator=gen, device="cuda", dtype=DTYPES[c["dtype"]])


def prepare(c, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    way, batch = c["way"], c["batch"]
    log2n = binding.benes_padded_log2n(c["n_elems"])
    perm, x = permutations(c, gen), payload(c, gen)
    s = {"way": way, "n": log2n, "n_elems": c["n_elems"], "batch": batch, "ebytes": BYTES[c["dtype"]],
         "perm": perm, "x": x}
    words = binding.benes_switch_words(log2n, batch)
    if way == "apply":
        s["bits"] = binding.route(perm)
    elif way == "padded":
        s["bits"] = torch.empty(words, dtype=torch.int32, device="cuda")
        s["out"] = torch.empty_like(x)
    elif way == "plan":
        s["bits"] = torch.empty(words, dtype=torch.int32, device="cuda")
        s["out"] = torch.empty_like(x)
        torch.cuda.synchronize()
        s["plan"] = binding.Plan(perm, log2n, batch, s["bits"], x, s["out"], s["ebytes"])
    elif way == "host":
        s["perm"], s["x"] = perm.cpu().pin_memory(), x.cpu().pin_memory()
        s["bits"] = torch.empty(words, dtype=torch.int32, pin_memory=True)
        s["out"] = torch.empty(x.shape, dtype=x.dtype, pin_memory=True)
    return s


def run(s):
    way = s["way"]
    if way == "calls":
        bits = binding.route(s["perm"])
        return {"bits": bits, "out": binding.apply(bits, s["x"])}
    if way == "apply":
        return {"out": binding.apply(s["bits"], s["x"])}
    if way == "padded":
        binding.benes_route_padded(s["perm"], s["n_elems"], s["batch"], s["bits"])
        binding.benes_apply_padded(s["bits"], s["x"], s["out"], s["ebytes"], s["n_elems"], s["batch"])
    elif way == "plan":
        s["plan"].launch()
    else:
        binding.benes_route_apply_host(s["perm"], s["x"], s["out"], s["ebytes"], s["n"], s["batch"], s["bits"])
    return {"bits": s["bits"], "out": s["out"]}


def work(c):
    """Permutation and payload read once, settings and routed payload written once (settings read for "apply")."""
    elems = c["n_elems"] * c["batch"]
    log2n = max(1, math.ceil(math.log2(c["n_elems"])))
    words = c["batch"] * (2 * log2n - 1) * max(1, (1 << log2n) // 64)
    perm = 0 if c["way"] == "apply" else 4 * elems
    return {"bytes": perm + 4 * words + 2 * elems * BYTES[c["dtype"]], "flops": 0}


def tolerance(c):
    """Settings are unique and payloads are only moved."""
    return "exact"

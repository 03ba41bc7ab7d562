"""What this library is used for, as measurable cases: packed bits in, packed bits out, through the C ABI's Python names.

A case fixes one call a user makes: which entry point, how many keys or blocks of which (n, m), in which
arithmetic. Keys and seeds are i.i.d. Bernoulli(0.5) bits, the model of reconciled QKD keys used by the tests
and the benchmark. Every output is the packed final keys (whole rows), so results compare as integers.
"""
import math

import torch

import paper_1809_07592_gb300 as pa

# The serving mix of the benchmark: block lengths and their weights.
SERVE_N = (1 << 18, 1_000_000, 1 << 22, 1 << 24)
SERVE_W = (0.4, 0.3, 0.2, 0.1)


def listed():
    return [
        # The smallest call: one short key on a cached seed. Launches and the guard's read-back are the cost.
        dict(name="tiny_fp32", kind="batch", n=5000, m=1500, keys=1, dtype="fp32_guard"),
        # The plain single block: one 131,072-bit key, 4:1 compression, double precision.
        dict(name="block_fp64", kind="batch", n=131072, m=32768, keys=1, dtype="fp64"),
        # A new Toeplitz seed for every block, as protocols that never reuse a seed need: seed upload and one key.
        dict(name="fresh_seed_fp32", kind="fresh", n=1 << 20, m=1 << 18, keys=1, dtype="fp32_guard"),
        # The modified Toeplitz hash on a small ragged batch: odd sizes, an odd number of keys, m not word aligned.
        dict(name="modified_ragged", kind="modified", n=100003, m=40001, keys=7, dtype="fp32_guard"),
        # DV-QKD batches on one cached seed, at the two ends of the compression range and both block lengths.
        dict(name="dv_1e6_tenth", kind="batch", n=1_000_000, m=100_000, keys=64, dtype="fp32_guard"),
        dict(name="dv_2p20_half", kind="batch", n=1 << 20, m=1 << 19, keys=64, dtype="fp32_guard"),
        # The same batch handed over in pinned host memory and taken back there (ingestion and egress).
        dict(name="dv_host", kind="host", n=1 << 20, m=1 << 18, keys=64, dtype="fp32_guard"),
        # The batch in the two wide arithmetics a caller can ask for.
        dict(name="dv_fp64", kind="batch", n=1_000_000, m=250_000, keys=64, dtype="fp64"),
        dict(name="dv_ntt64", kind="batch", n=1 << 20, m=1 << 18, keys=64, dtype="ntt64"),
        # The longest block: 2^27 bits to 2^24 with its seed spectrum resident.
        dict(name="long_fp32", kind="batch", n=1 << 27, m=1 << 24, keys=1, dtype="fp32_guard"),
        # An uneven batch, every block with its own length, compression and seed, replayed from its CUDA graph.
        dict(name="uneven_256", kind="uneven", blocks=256, lg_lo=16.0, lg_hi=24.0, mix=0, dtype="fp32_guard"),
        # A burst of 64 requests of the serving mix through the serving loop.
        dict(name="serving_64", kind="serving", blocks=64, mix=1, dtype="fp32_guard"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["batch", "batch", "batch", "fresh", "modified", "host", "long", "uneven", "serving"])
    if kind == "uneven":
        lo = rng.uniform(16.0, 20.0)
        return dict(kind=kind, blocks=_log_int(rng, 8, 192), lg_lo=lo, lg_hi=rng.uniform(lo + 1.0, 24.0),
                    mix=rng.randrange(1 << 20), dtype="fp32_guard")
    if kind == "serving":
        return dict(kind=kind, blocks=_log_int(rng, 8, 64), mix=rng.randrange(1 << 20), dtype="fp32_guard")
    if kind == "long":
        n = _log_int(rng, 1 << 22, 1 << 27)
        return dict(kind="batch", n=n, m=max(1, int(n * rng.uniform(0.05, 0.13))), keys=1, dtype="fp32_guard")
    n = _log_int(rng, 4000, 1 << 20)
    m = max(1, int(n * rng.uniform(0.05, 0.6)))
    dtype = rng.choice(["fp32_guard", "fp32_guard", "fp64", "ntt64"]) if kind == "batch" else "fp32_guard"
    keys = 1 if kind == "fresh" else _log_int(rng, 1, 40 if dtype != "fp32_guard" else 64)
    return dict(kind=kind, n=n, m=m, keys=keys, dtype=dtype)


def _sizes(case):
    """(n, m) of every block of an uneven batch or a serving burst."""
    g = torch.Generator().manual_seed(case["mix"])
    u = torch.rand(case["blocks"], 2, generator=g, dtype=torch.float64).tolist()
    out = []
    for a, b in u:
        if case["kind"] == "uneven":
            n = int(2.0 ** (case["lg_lo"] + (case["lg_hi"] - case["lg_lo"]) * a))
            m = int(n * (0.05 + 0.55 * b))
        else:
            i, acc = 0, SERVE_W[0]
            while a >= acc and i + 1 < len(SERVE_N):
                i += 1
                acc += SERVE_W[i]
            n = SERVE_N[i]
            m = int(n * (0.1 + 0.4 * b))
        out.append((n, max(1, m)))
    return out


def _words(bits):
    w = (bits + 63) // 64
    return w + (w & 1)  # even: every row 16-byte aligned


def _random_words(gen, *shape):
    return torch.randint(-(1 << 63), (1 << 63) - 1, shape, generator=gen, dtype=torch.int64, device="cuda")


def _seed_bits(case):
    return case["n"] - 1 if case["kind"] == "modified" else case["n"] + case["m"] - 1


def _inputs(case, seed):
    """Packed keys and seed of a shared-seed case; (keys, seeds) lists for blocks with their own."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if case["kind"] in ("uneven", "serving"):
        sizes = _sizes(case)
        return [(n, m, _random_words(gen, _words(n)), _random_words(gen, _words(n + m - 1))) for n, m in sizes]
    return _random_words(gen, case["keys"], _words(case["n"])), _random_words(gen, _words(_seed_bits(case)))


class _Handle:
    """An uneven batch or a server, released with the state that holds it."""

    def __init__(self, handle, destroy):
        self.handle, self._destroy = handle, destroy

    def __del__(self):
        try:
            self._destroy(self.handle)
        except Exception:
            pass


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("uneven", "serving"):
        data = _inputs(case, seed)
        # one buffer holds every block's final key, each at its own 16-byte aligned offset
        out = torch.zeros(sum(_words(m) for _, m, _, _ in data), dtype=torch.int64, device="cuda")
        blocks = [b + (o,) for b, o in zip(data, out.split([_words(m) for _, m, _, _ in data]))]
        torch.cuda.synchronize()  # the batch's and the server's own streams read these next
        if kind == "uneven":
            own = _Handle(pa.pa_uneven_create(blocks, case["dtype"], use_graph=True), pa.pa_uneven_destroy)
        else:
            own = _Handle(pa.pa_server_create(dtype=case["dtype"]), pa.pa_server_destroy)
        return dict(kind=kind, blocks=blocks, out=out, own=own)
    keys, sd = _inputs(case, seed)
    plan = pa.Plan(case["n"], case["m"], case["dtype"], modified=kind == "modified")
    plan.set_seed(sd)
    out = torch.zeros(case["keys"], _words(case["m"]), dtype=torch.int64, device="cuda")
    if kind == "host":
        keys, out = keys.cpu().pin_memory(), out.cpu().pin_memory()
    return dict(kind=kind, plan=plan, keys=keys, seed=sd, out=out)


def run(state):
    kind = state["kind"]
    if kind == "uneven":
        pa.pa_uneven_run(state["own"].handle, len(state["blocks"]))
        return state["out"]
    if kind == "serving":
        server = state["own"].handle
        tickets = [pa.pa_submit(server, *b) for b in state["blocks"]]
        for t in tickets:
            pa.pa_wait(server, t, 60000)
        return state["out"]
    plan, keys, out = state["plan"], state["keys"], state["out"]
    if kind == "host":
        pa.pa_hash_host(plan.handle, keys, keys.shape[0], keys.shape[1], out, out.shape[1])
        return out
    if kind == "fresh":
        plan.set_seed(state["seed"])
    plan.hash(keys, out)
    return out


def work(case):
    """Packed bits in and out; real transforms of the shortest cyclic length per key (and per seed that is not cached)."""
    if case["kind"] in ("uneven", "serving"):
        blocks = [(n, m, n + m - 1, 1, 1) for n, m in _sizes(case)]
    else:
        n, m = case["n"], case["m"]
        blocks = [(n, m, _seed_bits(case), case["keys"], 1 if case["kind"] == "fresh" else 0)]
    nbytes = flops = 0.0
    for n, m, length, keys, seeds in blocks:
        nbytes += (keys * (n + m) + seeds * length) / 8
        # a real transform is 2.5 N log2 N; each key takes one forward, one inverse and N/2 complex products
        flops += (2 * keys + seeds) * 2.5 * length * math.log2(max(length, 2)) + keys * 3.0 * length
    return {"bytes": nbytes, "flops": flops}


def _unpack(words, first, count):
    """Bits first .. first+count-1 of packed rows, as float64."""
    shifts = torch.arange(64, dtype=torch.int64, device=words.device)
    lo, hi = first // 64, (first + count + 63) // 64
    bits = ((words[..., lo:hi, None] >> shifts) & 1).flatten(-2)
    return bits[..., first - 64 * lo: first - 64 * lo + count].to(torch.float64)


def _pack(bits, nwords):
    """Rows of 0/1 float64 as packed int64 words, zero past the end."""
    m = bits.shape[-1]
    full = torch.zeros(*bits.shape[:-1], nwords * 64, dtype=torch.int64, device=bits.device)
    full[..., :m] = bits.to(torch.int64)
    shifts = torch.arange(64, dtype=torch.int64, device=bits.device)
    return (full.view(*bits.shape[:-1], nwords, 64) << shifts).sum(-1)


def _hash64(n, m, keys, sd, modified=False):
    """y_i = XOR_j s[i - j + cols - 1] x_j by one cyclic convolution in 64-bit floating point."""
    cols, first = (n - m, m) if modified else (n, 0)
    length = 1 << max(1, (cols + m - 2).bit_length())
    spec = torch.fft.rfft(_unpack(sd, 0, cols + m - 1), length)
    rows = []
    for k in keys:
        conv = torch.fft.irfft(torch.fft.rfft(_unpack(k, first, cols), length) * spec, length)
        y = torch.remainder(torch.round(conv[cols - 1: cols - 1 + m]), 2.0)
        if modified:
            y = torch.remainder(y + _unpack(k, 0, m), 2.0)
        rows.append(_pack(y, _words(m)))
    return torch.stack(rows)


def exact(case, seed):
    if case["kind"] in ("uneven", "serving"):
        return torch.cat([_hash64(n, m, k[None], s)[0] for n, m, k, s in _inputs(case, seed)])
    keys, sd = _inputs(case, seed)
    y = _hash64(case["n"], case["m"], keys, sd, case["kind"] == "modified")
    return y.cpu() if case["kind"] == "host" else y

"""What the performance of this library is measured on.

Every case is work a program has the library do through the public binding
(`paper_2402_09481_gb300.native`): single extractions of the three kinds from
the shortest keys to the two-source example of 2^30 bits, the two-source ->
seeded composition, the host-buffer call, the planned batch, many inputs under
one seed, the request server, the Von Neumann filter and Trevisan's one-bit
step.  Sizes are the workloads of the benchmark and the tests of this
repository, with ragged ones between them.  All arithmetic is on packed bits:
outputs are int64 words (and an int64 length for Von Neumann).
"""

import math

import numpy as np
import torch

from paper_2402_09481_gb300 import native

TOEPLITZ, CIRCULANT, DODIS = 0, 1, 2


def listed():
    return [
        # one short key block: a latency-bound call a protocol makes per frame
        dict(name="toeplitz_4k", what="single", kind=TOEPLITZ, n=4096, m=2048),
        # the benchmark's short extraction (input 2^16, output 2^15)
        dict(name="toeplitz_64k", what="single", kind=TOEPLITZ, n=65536, m=32768),
        # a ragged block of an ordinary size (neither length a multiple of 64)
        dict(name="toeplitz_300k", what="single", kind=TOEPLITZ, n=300007, m=150001),
        # the benchmark's default extraction: n + 1 the smallest admissible prime above 2^24
        dict(name="circulant_16m", what="single", kind=CIRCULANT, n=16777258, m=8388629),
        # the benchmark's two-source extraction, a biased first source
        dict(name="dodis_1g", what="single", kind=DODIS, n=1073741789, m=429496715),
        # two-source extraction whose output seeds a second extraction of the weak seed
        dict(name="compose_4m", what="compose", n1=4194389, m1=2000003, n2=1200000, m2=800003),
        # privacy amplification of a distilled key held in host memory (the QKD
        # example's output rate at a quarter of its length): copies included
        dict(name="host_qkd", what="host", kind=TOEPLITZ, n=434500000, m=10344566),
        # the benchmark's batch: 4096 blocks of log-uniform length, own seeds
        dict(name="batch_4096", what="batch", count=4096, lo=10.0, hi=22.0),
        # the benchmark's shared-seed product
        dict(name="shared_seed_64k", what="shared", n=4096, m=2048, count=65536),
        # a burst of mixed requests to the server
        dict(name="served_48", what="served", count=48, lo=12.0, hi=23.0),
        # debiasing of a raw generator's bits (the QRNG example's input length)
        dict(name="von_neumann_6g", what="vn", n=6500000000),
        # Trevisan's one-bit step at the benchmark's size
        dict(name="trevisan_1m", what="trevisan", n=1 << 20, m=1 << 16, l=121),
    ]


# --------------------------------------------------------------------------- #
# admissible lengths: primes with 2 as a primitive root


def _factors(v):
    out, p = [], 2
    while p * p <= v:
        if v % p == 0:
            out.append(p)
            while v % p == 0:
                v //= p
        p += 1 if p == 2 else 2
    if v > 1:
        out.append(v)
    return out


def _admissible(P):
    if P < 3 or P % 2 == 0 or pow(2, P - 1, P) != 1:
        return False
    if any(P % p == 0 for p in range(3, math.isqrt(P) + 1, 2)):
        return False
    return all(pow(2, (P - 1) // f, P) != 1 for f in _factors(P - 1))


def _next_admissible(v):
    v = max(v, 3)
    while not _admissible(v):
        v += 1
    return v


def _logint(rng, lo, hi):
    return int(2.0 ** rng.uniform(lo, hi))


def draw(rng):
    what = rng.choice(["single", "single", "single", "single", "single", "compose", "host", "batch", "shared",
                       "served", "vn", "trevisan"])
    if what in ("single", "host"):
        kind = rng.choice([TOEPLITZ, CIRCULANT, DODIS])
        n = _logint(rng, 10, 27.5)
        if kind == CIRCULANT:
            n = _next_admissible(n + 1) - 1
        elif kind == DODIS:
            n = _next_admissible(n)
        return dict(what=what, kind=kind, n=n, m=max(1, int(n * rng.uniform(0.02, 0.6))))
    if what == "compose":
        n1 = _next_admissible(_logint(rng, 12, 23))
        m1 = int(n1 * rng.uniform(0.3, 0.6))
        n2 = int(m1 * rng.uniform(0.4, 0.6))
        return dict(what=what, n1=n1, m1=m1, n2=n2, m2=int((m1 - n2) * rng.uniform(0.5, 1.0)))
    if what == "batch":
        lo = rng.uniform(10, 14)
        return dict(what=what, count=_logint(rng, 5, 10), lo=lo, hi=lo + rng.uniform(2, 8))
    if what == "shared":
        n = _logint(rng, 8, 13)
        return dict(what=what, n=n, m=max(1, int(n * rng.uniform(0.1, 0.8))), count=_logint(rng, 8, 15))
    if what == "served":
        lo = rng.uniform(10, 14)
        return dict(what=what, count=rng.randint(4, 64), lo=lo, hi=lo + rng.uniform(2, 8))
    if what == "vn":
        return dict(what=what, n=_logint(rng, 18, 32))
    l = rng.randint(40, 160)
    return dict(what=what, n=_logint(rng, 12, 20), m=_logint(rng, 7, 16 if l <= 120 else 15), l=l)


# --------------------------------------------------------------------------- #
# inputs, from the seed alone


def _words(bits):
    return (bits + 63) // 64


def _rand(gen, bits, biased=False):
    """Packed random bits on the GPU; biased: P(1) = 3/4."""
    def r():
        return torch.randint(-2 ** 63, 2 ** 63 - 1, (max(1, _words(bits)),), dtype=torch.int64, device="cuda",
                             generator=gen)
    w = r() | r() if biased else r()
    return w


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _ybits(kind, n, m):
    return n + m - 1 if kind == TOEPLITZ else (n + 1 if kind == CIRCULANT else n)


def _pair(gen, kind, n, m):
    return _rand(gen, n, biased=kind == DODIS), _rand(gen, _ybits(kind, n, m))


def _lengths(case, seed, kinds):
    """(kind, n, m) of a batch or a burst: lengths log-uniform, outputs half as long."""
    rng = np.random.default_rng(seed)
    u = rng.uniform(case["lo"], case["hi"], case["count"])
    out = []
    for j in range(case["count"]):
        kind, n = kinds[j % len(kinds)], int(2.0 ** u[j])
        if kind == CIRCULANT:
            n = _next_admissible(n + 1) - 1
        elif kind == DODIS:
            n = _next_admissible(n)
        out.append((kind, n, n // 2))
    return out


BATCH_KINDS = [TOEPLITZ]
SERVED_KINDS = [TOEPLITZ, TOEPLITZ, CIRCULANT, DODIS]


def _many(case, seed, kinds):
    gen = _gen(seed)
    spec = _lengths(case, 12345, kinds)  # the lengths belong to the case, the bits to the seed
    return [(kind, n, m, *_pair(gen, kind, n, m)) for kind, n, m in spec]


def _items(case, seed, kinds):
    """Descriptors whose outputs lie back to back in one buffer, and that buffer."""
    many = _many(case, seed, kinds)
    zs = torch.zeros(sum(_words(m) for _, _, m, _, _ in many), dtype=torch.int64, device="cuda")
    items, at = [], 0
    for k, n, m, x, y in many:
        items.append((k, n, m, x, y, zs[at:at + _words(m)]))
        at += _words(m)
    return items, zs


def prepare(case, seed):
    what = case["what"]
    st = dict(case=case, ctx=native.Context(0))
    gen = _gen(seed)
    if what == "single":
        st["x"], st["y"] = _pair(gen, case["kind"], case["n"], case["m"])
        st["z"] = torch.zeros(_words(case["m"]), dtype=torch.int64, device="cuda")
    elif what == "compose":
        st["x"], st["y"] = _pair(gen, DODIS, case["n1"], case["m1"])
        st["z"] = torch.zeros(_words(case["m1"] + case["m2"]), dtype=torch.int64, device="cuda")
    elif what == "host":
        x, y = _pair(gen, case["kind"], case["n"], case["m"])
        st["x"], st["y"] = x.cpu().pin_memory(), y.cpu().pin_memory()
        st["z"] = torch.zeros(_words(case["m"]), dtype=torch.int64).pin_memory()
    elif what == "batch":
        st["items"], st["zs"] = _items(case, seed, BATCH_KINDS)
        st["batch"] = st["ctx"].batch(st["items"], autotune=True)
    elif what == "served":
        st["items"], st["zs"] = _items(case, seed, SERVED_KINDS)
        torch.cuda.synchronize()  # the server's streams read the inputs
        st["ctx"].server_start()
    elif what == "shared":
        st["y"] = _rand(gen, case["n"] + case["m"] - 1)
        st["X"] = _rand(gen, _words(case["n"]) * 64 * case["count"])
        st["Z"] = torch.zeros(_words(case["m"]) * case["count"], dtype=torch.int64, device="cuda")
    elif what == "vn":
        st["x"] = _rand(gen, case["n"])
        st["z"] = torch.zeros(max(1, _words(case["n"] // 2)), dtype=torch.int64, device="cuda")
        st["mo"] = torch.zeros(1, dtype=torch.int64, device="cuda")
    else:
        st["x"] = _rand(gen, case["n"])
        st["s"] = _rand(gen, 2 * case["l"] * case["m"])
        st["z"] = torch.zeros(_words(case["m"]), dtype=torch.int64, device="cuda")
    return st


def run(st):
    case, ctx = st["case"], st["ctx"]
    what = case["what"]
    if what == "single":
        n, m = case["n"], case["m"]
        if case["kind"] == TOEPLITZ:
            return ctx.toeplitz(st["x"], n, st["y"], m, st["z"])
        if case["kind"] == CIRCULANT:
            return ctx.circulant(st["x"], n, st["y"], m, st["z"])
        return ctx.dodis(st["x"], st["y"], n, m, st["z"])
    if what == "compose":
        return ctx.compose(DODIS, st["x"], case["n1"], st["y"], case["m1"], TOEPLITZ, case["n2"], case["m2"],
                           st["z"])
    if what == "host":
        ctx.extract_host(case["kind"], st["x"], case["n"], st["y"], case["m"], st["z"])
        return st["z"]
    if what == "batch":
        st["batch"].launch()
        return st["zs"]
    if what == "served":
        tickets = [ctx.submit(*it) for it in st["items"]]
        for t in tickets:
            ctx.poll(t, 60.0)
        return st["zs"]
    if what == "shared":
        return ctx.toeplitz_shared_seed(st["y"], case["n"], case["m"], st["X"], case["count"], st["Z"])
    if what == "vn":
        return list(ctx.von_neumann(st["x"], case["n"], st["z"], st["mo"]))
    return ctx.trevisan_rsh(st["x"], case["n"], case["l"], st["s"], case["m"], st["z"])


# --------------------------------------------------------------------------- #
# what a pass cannot do without


def _extraction(kind, n, m):
    """Bits in and out once; operations of the convolution by transforms."""
    L = n + m
    return (n + _ybits(kind, n, m) + m) / 8, 3 * L * math.log2(max(L, 2))


def work(case):
    what = case["what"]
    if what in ("single", "host"):
        b, f = _extraction(case["kind"], case["n"], case["m"])
    elif what == "compose":
        b1, f1 = _extraction(DODIS, case["n1"], case["m1"])
        b2, f2 = _extraction(TOEPLITZ, case["n2"], case["m2"])
        b, f = b1 + b2, f1 + f2
    elif what in ("batch", "served"):
        kinds = BATCH_KINDS if what == "batch" else SERVED_KINDS
        parts = [_extraction(*spec) for spec in _lengths(case, 12345, kinds)]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    elif what == "shared":
        b = (case["n"] + case["m"]) * case["count"] / 8
        f = 2.0 * case["n"] * case["m"] * case["count"]
    elif what == "vn":
        b, f = case["n"] / 8 + case["n"] / 32, case["n"]
    else:
        chunks = -(-case["n"] // case["l"])
        b = (case["n"] + 2 * case["l"] * case["m"] + case["m"]) / 8
        f = 2.0 * chunks * case["l"] ** 2 * case["m"]
    return {"bytes": float(b), "flops": float(f)}


# --------------------------------------------------------------------------- #
# the definitions, in 64-bit numbers


def _bits(w, n):
    """n bits of packed words as a uint8 tensor."""
    sh = torch.arange(64, device=w.device, dtype=torch.int64)
    out = torch.empty(w.numel() * 64, dtype=torch.uint8, device=w.device)
    step = 1 << 22
    for i in range(0, w.numel(), step):
        out[i * 64:(i + step) * 64] = ((w[i:i + step, None] >> sh) & 1).to(torch.uint8).reshape(-1)
    return out[:n]


def _pack(b):
    """uint8 bits to int64 words, the last one padded with 0."""
    k = _words(b.numel())
    out = torch.zeros(k, dtype=torch.int64, device=b.device)
    sh = torch.arange(64, device=b.device, dtype=torch.int64)
    step = 1 << 22
    for i in range(0, k, step):
        part = b[i * 64:(i + step) * 64]
        rows = _words(part.numel())
        buf = torch.zeros(rows * 64, dtype=torch.uint8, device=b.device)
        buf[:part.numel()] = part
        out[i:i + rows] = (buf.reshape(rows, 64).to(torch.int64) << sh).sum(1)
    return out


def _extract_bits(kind, xb, n, yb, m):
    """Output bits from the displayed matrices, by a real convolution in 64 bits."""
    if kind == TOEPLITZ:      # z_i = sum_j y[(i - j) mod (n + m - 1)] x_j
        a, b = xb, torch.roll(yb, n - 1)
        lo = n - 1            # b[k] = y[k - (n - 1)]: z_i = (x * b)[n - 1 + i]
    else:                     # z_i = sum_j x'[(j - i) mod P] y_j, x' = [x, 0] for Circulant
        P = n + 1 if kind == CIRCULANT else n
        xp = torch.zeros(P, dtype=torch.uint8, device=xb.device)
        xp[:n] = xb
        a, b = torch.flip(xp, (0,)), torch.cat([yb, yb[:m - 1]]) if m > 1 else yb
        lo = P - 1
    L = 1 << (a.numel() + b.numel() - 1).bit_length()
    if L >> 1 >= b.numel():   # wrapped terms stay below the window
        L >>= 1
    fa = torch.fft.rfft(a.double(), L)
    fa *= torch.fft.rfft(b.double(), L)
    c = torch.fft.irfft(fa, L)[lo:lo + m]
    return (torch.round(c).to(torch.int64) & 1).to(torch.uint8)


def _extract(kind, x, n, y, m):
    return _extract_bits(kind, _bits(x, n), n, _bits(y, _ybits(kind, n, m)), m)


def exact(case, seed):
    what = case["what"]
    gen = _gen(seed)
    if what in ("single", "host"):
        if case["n"] + case["m"] > 1 << 28:
            return None       # minutes in 64-bit transforms of this length
        x, y = _pair(gen, case["kind"], case["n"], case["m"])
        z = _pack(_extract(case["kind"], x, case["n"], y, case["m"]))
        return z.cpu() if what == "host" else z
    if what == "compose":
        x, y = _pair(gen, DODIS, case["n1"], case["m1"])
        s = _extract(DODIS, x, case["n1"], y, case["m1"])
        n2, m2 = case["n2"], case["m2"]
        t = _extract_bits(TOEPLITZ, _bits(y, n2), n2, s[:n2 + m2 - 1], m2)
        return _pack(torch.cat([s, t]))
    if what in ("batch", "served"):
        kinds = BATCH_KINDS if what == "batch" else SERVED_KINDS
        return torch.cat([_pack(_extract(k, x, n, y, m)) for k, n, m, x, y in _many(case, seed, kinds)])
    if what == "shared":
        n, m, count = case["n"], case["m"], case["count"]
        yb = _bits(_rand(gen, n + m - 1), n + m - 1)
        X = _rand(gen, _words(n) * 64 * count)
        idx = (torch.arange(m, device="cuda")[:, None] - torch.arange(n, device="cuda")[None, :]) % (n + m - 1)
        T = yb[idx].double()
        wn, wm = _words(n), _words(m)
        out = torch.zeros(count, wm, dtype=torch.int64, device="cuda")
        step = 4096
        for c in range(0, count, step):
            cc = min(step, count - c)
            xb = _bits(X[c * wn:(c + cc) * wn], cc * wn * 64).reshape(cc, wn * 64)[:, :n].double()
            zb = (torch.round(xb @ T.T).to(torch.int64) & 1).to(torch.uint8)
            pad = torch.zeros(cc, wm * 64, dtype=torch.uint8, device="cuda")
            pad[:, :m] = zb
            out[c:c + cc] = _pack(pad.reshape(-1)).reshape(cc, wm)
        return out.reshape(-1)
    if what == "vn":
        n = case["n"]
        x = _rand(gen, n)
        parts, step = [], 1 << 27
        for i in range(0, n - 1, step):
            b = _bits(x[i // 64:(i + step) // 64 + 1], min(step, n - i))
            b = b[:b.numel() // 2 * 2].reshape(-1, 2)
            parts.append(b[b[:, 0] != b[:, 1], 0])
        bits = torch.cat(parts)
        z = torch.zeros(max(1, _words(n // 2)), dtype=torch.int64, device="cuda")
        z[:_words(bits.numel())] = _pack(bits)
        return [z, torch.tensor([bits.numel()], dtype=torch.int64, device="cuda")]
    return None               # the field arithmetic takes minutes outside a kernel

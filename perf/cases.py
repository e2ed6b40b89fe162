"""What this framework is timed on: its public entry points at the sizes its users have.

Every case is one call sequence a program makes (build a graph and take it out
sorted, add reads to a held graph, assemble contigs, size tables, train the
sizing network).  Inputs are synthetic read sets made on the GPU from a seed:
uniform genomes (with 1 kb repeats where a case says so), reads at uniform
positions, independent substitution errors -- the distributions of the
package's own generator, drawn with torch so that 20 million reads take well
under a second.
"""

import math

import numpy as np
import torch

from paper_2401_02756_gb300 import dbg

DEV = "cuda"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _reads(genome, cov, read, err, k, repeats=False, ragged=False, **more):
    return dict(genome=genome, cov=float(cov), read=read, err=float(err), k=k, repeats=repeats,
                ragged=ragged, **more)


def listed():
    return [
        # the smallest request: a 10 kb error-free amplicon or plasmid, where
        # launches and synchronisations are everything
        dict(name="build_10kb_k21", do="build", **_reads(10_000, 10, 100, 0.0, 21)),
        # one ordinary sample of the batched workload, built alone (its table is
        # below the binned path's size: the direct insert)
        dict(name="build_300kb_k21", do="build", **_reads(300_000, 35, 150, 0.005, 21)),
        # a bacterial genome at 50x with 1 % errors, the size of the paper's E. coli runs
        dict(name="build_5mbp_k31", do="build", **_reads(5_000_000, 50, 150, 0.01, 31)),
        # the largest: 100 Mbp with 5 % repeats at 30x, the sorted graph in kept device buffers
        dict(name="build_100mbp_k31", do="build",
             **_reads(100_000_000, 30, 150, 0.005, 31, repeats=True)),
        # the paper's default k (128-bit keys) on the bacterial genome, reads of uneven length
        dict(name="build_5mbp_k51", do="build", **_reads(5_000_000, 50, 150, 0.01, 51, ragged=True)),
        # many samples at once: the batched build, then every graph out through caller memory
        dict(name="batch_24", do="batch", items=24, genome_lo=50_000, genome_hi=2_000_000,
             cov_lo=10.0, cov_hi=60.0, read=150, err=0.005),
        # reads that arrive in four lots: reset, then four inserts into the held graph
        dict(name="insert_4lots_2mbp_k31", do="insert", lots=4,
             **_reads(2_000_000, 30, 150, 0.005, 31)),
        # one request of the serving loop: reads in pinned host memory, the
        # sorted graph back in pinned host memory
        dict(name="request_1mbp_k31", do="host", **_reads(1_000_000, 30, 150, 0.005, 31)),
        # assembly of the bacterial genome: build, normalize by the coverage, contigs
        dict(name="assemble_5mbp_k31", do="assemble", **_reads(5_000_000, 50, 150, 0.01, 31)),
        # assembly of a small error-free genome: few, long contigs
        dict(name="assemble_50kb_k21", do="assemble", **_reads(50_000, 30, 100, 0.0, 21)),
        # table sizes for 64 samples before they are built: sketches and the network
        dict(name="size_64", do="size", items=64, genome_lo=50_000, genome_hi=2_000_000,
             cov_lo=10.0, cov_hi=60.0, read=150, err=0.005),
        # one training step of the sizing network at its training batch
        dict(name="train_256", do="train", batch=256),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["build", "build", "build", "wide", "batch", "insert", "host", "assemble",
                     "clean", "size", "train"])
    ragged = rng.random() < 0.4
    read = rng.choice([75, 100, 101, 150, 151, 250])
    err = rng.choice([0.0, 0.001, 0.005, 0.01])
    cov = round(rng.uniform(8, 55), 1)
    if do == "build":
        return dict(do="build", **_reads(_log_uniform(rng, 5_000, 30_000_000), cov, read, err,
                                         rng.choice([11, 15, 21, 25, 27, 31, 32]),
                                         repeats=rng.random() < 0.5, ragged=ragged))
    if do == "wide":
        return dict(do="build", **_reads(_log_uniform(rng, 5_000, 5_000_000), cov, max(read, 100),
                                         err, rng.choice([33, 41, 51, 63, 64]), ragged=ragged))
    if do == "insert":
        return dict(do="insert", lots=rng.randint(2, 6),
                    **_reads(_log_uniform(rng, 50_000, 8_000_000), cov, read, err,
                             rng.choice([15, 21, 31]), ragged=ragged))
    if do == "host":
        return dict(do="host", **_reads(_log_uniform(rng, 50_000, 4_000_000), cov, read, err,
                                        rng.choice([21, 31, 51]), ragged=ragged))
    if do == "assemble":
        return dict(do="assemble", **_reads(_log_uniform(rng, 50_000, 5_000_000),
                                            round(rng.uniform(20, 50), 1), max(read, 100),
                                            rng.choice([0.001, 0.005, 0.01]), rng.choice([21, 25, 31])))
    if do == "clean":
        return dict(do="assemble", **_reads(_log_uniform(rng, 5_000, 70_000),
                                            round(rng.uniform(15, 40), 1), max(read, 100), 0.0,
                                            rng.choice([21, 31])))
    if do in ("batch", "size"):
        return dict(do=do, items=rng.randint(3, 30 if do == "batch" else 100), genome_lo=50_000,
                    genome_hi=2_000_000, cov_lo=10.0, cov_hi=rng.choice([30.0, 60.0]), read=read,
                    err=0.005)
    return dict(do="train", batch=_log_uniform(rng, 16, 1000))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 2654435761 % (1 << 62) + 12345)
    return g


def _genome(n, repeats, gen):
    g = torch.randint(0, 4, (n,), dtype=torch.uint8, device=DEV, generator=gen)
    copies = n // 20_000  # 1 kb copies over 5 % of the genome
    if repeats and copies >= 2:
        families = max(1, copies // 15)
        segment = torch.randint(0, 4, (families, 1000), dtype=torch.uint8, device=DEV, generator=gen)
        which = torch.randint(0, families, (copies,), device=DEV, generator=gen)
        where = torch.randperm(n // 1000, device=DEV, generator=gen)[:copies]
        text = segment[which]
        mutated = torch.rand(text.shape, device=DEV, generator=gen) < 0.001
        text = (text + mutated.to(torch.uint8)) & 3
        g[:n // 1000 * 1000].view(-1, 1000)[where] = text
    return g


def _n_reads(genome, cov, read):
    return max(1, int(round(cov * genome / read)))


def _read_set(genome, cov, read, err, repeats, ragged, gen):
    """(packed uint8, offsets int64) on the GPU."""
    text = _genome(genome, repeats, gen)
    n = _n_reads(genome, cov, read)
    longest = min(genome, read + read // 2 if ragged else read)
    if ragged:  # lengths uniform about the mean, a few shorter than any k
        lens = torch.randint(read // 2, longest + 1, (n,), device=DEV, generator=gen)
        lens[::997] = 9
    else:
        lens = torch.full((n,), longest, device=DEV, dtype=torch.int64)
    starts = (torch.rand(n, device=DEV, dtype=torch.float64, generator=gen)
              * (genome - lens + 1)).to(torch.int64)
    offsets = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(lens, 0, out=offsets[1:])
    total = int(offsets[-1])
    codes = torch.zeros((total + 3) // 4 * 4, dtype=torch.uint8, device=DEV)
    step = 1 << 19
    for r0 in range(0, n, step):
        r1 = min(n, r0 + step)
        b0, b1 = int(offsets[r0]), int(offsets[r1])
        if ragged:
            shift = torch.repeat_interleave(starts[r0:r1] - offsets[r0:r1], lens[r0:r1],
                                            output_size=b1 - b0)
            c = text[torch.arange(b0, b1, device=DEV) + shift]
        else:
            c = text[(starts[r0:r1, None] + torch.arange(longest, device=DEV)).view(-1)]
        if err > 0:
            wrong = torch.rand(c.numel(), device=DEV, generator=gen) < err
            by = torch.randint(1, 4, (c.numel(),), dtype=torch.uint8, device=DEV, generator=gen)
            c = (c + by * wrong) & 3
        codes[b0:b1] = c
    c = codes.view(-1, 4)
    packed = c[:, 0] | (c[:, 1] << 2) | (c[:, 2] << 4) | (c[:, 3] << 6)
    return packed, offsets


def _vertices(case):
    """Expected distinct vertices, a few per cent high: what a program that
    knows its genome size and error rate sizes its table by."""
    m = case["k"] - 1
    n = _n_reads(case["genome"], case["cov"], case["read"])
    windows = n * max(0, case["read"] - m + 1)
    wrong = windows * (1.0 - (1.0 - case["err"]) ** m)
    return int(min(case["genome"] + wrong + 64, 4.0 ** min(m, 40) + 64, windows + n * m + 64))


def _positions(case):
    n = _n_reads(case["genome"], case["cov"], case["read"])
    return n * max(0, case["read"] - case["k"] + 2)


def _samples(case):
    """The batched workload's samples: genome sizes log-uniform, coverage uniform, k 21 or 31."""
    u = np.random.RandomState(case["items"]).random_sample((case["items"], 3))
    out = []
    for a, b, c in u:
        genome = int(case["genome_lo"] * (case["genome_hi"] / case["genome_lo"]) ** a)
        out.append(_reads(genome, case["cov_lo"] + b * (case["cov_hi"] - case["cov_lo"]),
                          case["read"], case["err"], 21 if c < 0.5 else 31))
    return out


def _one(case, gen):
    return _read_set(case["genome"], case["cov"], case["read"], case["err"], case["repeats"],
                     case["ragged"], gen)


def _out_buffers(rows, k):
    return (torch.empty((rows, 2) if k > 32 else rows, dtype=torch.int64, device=DEV),
            torch.empty((rows, 4), dtype=torch.int32, device=DEV))


def prepare(case, seed):
    gen = _generator(seed)
    do = case["do"]
    s = {"do": do, "case": case}
    if do in ("build", "insert", "host", "assemble"):
        packed, offsets = _one(case, gen)
        k, want = case["k"], _vertices(case)
        if case["genome"] * case["cov"] > 5e8:
            torch.cuda.empty_cache()  # the generator's temporaries
        g = dbg.Graph(k, max(64, int(want * 1.5)))
        if k <= 31:
            g.reserve_events(_positions(case) + _positions(case) // 50)
        s.update(graph=g, packed=packed, offsets=offsets)
        if do in ("build", "insert"):
            s["out"] = _out_buffers(want + want // 16, k)
        if do == "insert":
            n = offsets.numel() - 1
            cut = [n * i // case["lots"] for i in range(case["lots"] + 1)]
            s["lots"] = [offsets[a:b + 1].clone() for a, b in zip(cut, cut[1:])]
        elif do == "host":
            s["packed"], s["offsets"] = packed.cpu().pin_memory(), offsets.cpu().pin_memory()
            rows = want + want // 16
            s["out"] = (torch.zeros((rows, 2) if k > 32 else rows, dtype=torch.int64,
                                    pin_memory=True).numpy(),
                        torch.zeros((rows, 4), dtype=torch.int32, pin_memory=True).numpy())
        elif do == "assemble":
            edges = float((offsets.diff() - k + 1).clamp(min=0).sum())
            s["divisor"] = max(1.0, edges / case["genome"])
            s["text"] = np.zeros(6 * case["genome"] + 65536, dtype=np.uint8)
    elif do == "batch":
        s["items"], s["out"], most = [], [], 0
        for c in _samples(case):
            packed, offsets = _one(c, gen)
            want = _vertices(c)
            g = dbg.Graph(c["k"], int(want * 1.5))
            g.reserve_events(_positions(c))
            rows = want + want // 16
            most = max(most, dbg.export_scratch_bytes(c["k"], rows, g.info()["n_slots"]))
            s["items"].append((g, packed, offsets))
            s["out"].append(_out_buffers(rows, c["k"]))
        s["scratch"] = torch.empty(most, dtype=torch.uint8, device=DEV)
    elif do == "size":
        n = case["items"]
        samples = [(c["k"],) + _one(c, gen) for c in _samples(case)]
        regs = torch.empty(n, dbg.SKETCH_REGISTERS + 1, dtype=torch.int32, device=DEV)
        s.update(items=[(k, p, o, regs[i]) for i, (k, p, o) in enumerate(samples)], regs=regs,
                 params=_network(gen)[0], x=torch.empty(n, dbg.MLP_INPUTS, device=DEV),
                 y=torch.empty(n, device=DEV), work=torch.empty(dbg.mlp_work_floats(n), device=DEV))
    else:
        b = case["batch"]
        params, m, v = _network(gen)
        x, target = _training_rows(b, gen)
        s.update(params=params, m=m, v=v, x=x, target=target, grads=torch.zeros_like(params),
                 loss=torch.zeros(1, device=DEV), step=200,
                 work=torch.empty(dbg.mlp_work_floats(b), device=DEV))
    return s


def _network(gen):
    """Weights of the network's scale, with Adam moments as some way into training."""
    n1, h = dbg.MLP_INPUTS, dbg.MLP_HIDDEN
    p = torch.zeros(dbg.MLP_PARAMS, device=DEV)
    u = torch.rand(dbg.MLP_PARAMS, device=DEV, generator=gen) * 2 - 1
    a, b, c, d = h * n1, h * n1 + h, h * n1 + h + h * h, h * n1 + 2 * h + h * h
    p[:a] = u[:a] * math.sqrt(6 / n1)
    p[a:b] = u[a:b] * 0.1
    p[b:c] = u[b:c] * math.sqrt(6 / h)
    p[c:d] = u[c:d] * 0.1
    p[d:] = u[d:] * math.sqrt(6 / h)
    m = torch.randn(dbg.MLP_PARAMS, device=DEV, generator=gen) * 1e-2
    v = torch.rand(dbg.MLP_PARAMS, device=DEV, generator=gen) * 1e-3 + 1e-4
    return p, m, v


def _training_rows(b, gen):
    """Register rows of sketches of n distinct keys (each the maximum of n / 1024
    geometric draws), n log-uniform over the training range, and ln n."""
    ln_n = torch.rand(b, device=DEV, generator=gen) * math.log(15e6 / 9.6e4) + math.log(9.6e4)
    u = torch.rand(b, dbg.MLP_INPUTS, device=DEV, dtype=torch.float64, generator=gen)
    per = torch.exp(ln_n.double())[:, None] / dbg.MLP_INPUTS
    regs = torch.floor(-torch.log2(-torch.log(u.clamp(min=1e-12)) / per)).clamp(1, 54) + 1
    return (regs / 64).float(), ln_n


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _sorted(out, export, *more):
    """The sorted graph in kept buffers; the rows past its vertices are zeroed,
    since the export leaves them as it likes."""
    keys, counts = out
    n = export(keys, counts, *more)
    keys[n:].zero_()
    counts[n:].zero_()
    return [keys, counts]


def run(s):
    do = s["do"]
    if do == "build":
        g = s["graph"]
        g.build(s["packed"], s["offsets"])
        return _sorted(s["out"], g.export_into)
    if do == "insert":
        g = s["graph"]
        g.reset()
        for offsets in s["lots"]:
            g.insert(s["packed"], offsets)
        return _sorted(s["out"], g.export_into) + list(g.stats())
    if do == "host":
        g = s["graph"]
        g.build_host(s["packed"], s["offsets"])
        keys, _ = g.export(out=s["out"])
        return list(s["out"]) + [len(keys)]
    if do == "assemble":
        g = s["graph"]
        g.build(s["packed"], s["offsets"])
        g.normalize(s["divisor"])
        contigs = "\n".join(g.contigs()).encode()
        s["text"][:len(contigs)] = np.frombuffer(contigs, dtype=np.uint8)
        return s["text"]
    if do == "batch":
        dbg.build_batch(s["items"])
        out = []
        for (g, _, _), (keys, counts) in zip(s["items"], s["out"]):
            out += _sorted((keys, counts), g.export_with, s["scratch"])
        return out
    if do == "size":
        n = len(s["items"])
        dbg.sketch_batch(s["items"])
        dbg.mlp_features(s["regs"], s["x"], n)
        dbg.mlp_forward(s["params"], s["x"], s["y"], s["work"], batch=n)
        return s["y"], s["regs"]
    s["step"] += 1
    dbg.mlp_train_step(s["params"], s["grads"], s["m"], s["v"], s["step"], 1e-3, s["x"],
                       s["target"], s["work"], loss=s["loss"])
    return {"params": s["params"], "grads": s["grads"], "m": s["m"], "v": s["v"],
            "loss": s["loss"]}


def work(case):
    """Inputs read once and results written once; the multiply-adds of the network."""
    do, flops = case["do"], 0.0
    if do == "train":
        p, b = dbg.MLP_PARAMS, case["batch"]
        # weights, gradients and both moments (three read, four written), the rows
        return {"bytes": 4.0 * (7 * p + b * (dbg.MLP_INPUTS + 1)), "flops": 6.0 * p * b}

    def of(c, rows):
        n = _n_reads(c["genome"], c["cov"], c["read"])
        return n * c["read"] / 4 + 8 * n + rows * _vertices(c) * (32 if c["k"] > 32 else 24)

    if do in ("batch", "size"):
        bytes_ = sum(of(c, do == "batch") for c in _samples(case))
        if do == "size":
            bytes_ += 4.0 * dbg.MLP_PARAMS + case["items"] * 4.0 * (dbg.MLP_INPUTS + 2)
            flops = 2.0 * dbg.MLP_PARAMS * case["items"]
        return {"bytes": bytes_, "flops": flops}
    if do == "assemble":
        return {"bytes": of(case, 0) + 1.2 * case["genome"], "flops": 0.0}
    return {"bytes": of(case, 1), "flops": 0.0}


# ---------------------------------------------------------------------------
# what the computed numbers are in 64 bits (the graphs are whole numbers)
# ---------------------------------------------------------------------------

def _layers(p):
    n1, h = dbg.MLP_INPUTS, dbg.MLP_HIDDEN
    at, out = 0, []
    for shape in ((h, n1), (h,), (h, h), (h,), (h,), (1,)):
        n = math.prod(shape)
        out.append(p[at:at + n].view(shape))
        at += n
    return out


def _forward(p, x):
    w1, b1, w2, b2, w3, b3 = _layers(p)
    h1 = torch.relu(x @ w1.T + b1)
    return torch.relu(h1 @ w2.T + b2) @ w3 + b3


_M1, _M2, _SALT = (c - (1 << 64) if c >> 63 else c for c in
                   (0xff51afd7ed558ccd, 0xc4ceb9fe1a85ec53, 0x9E3779B97F4A7C15))


def _shift(x, n):  # logical right shift of int64
    return (x >> n) & ((1 << (64 - n)) - 1)


def _registers(k, packed, offsets):
    """HyperLogLog registers of a read set's (k-1)-base windows."""
    m = k - 1
    codes = torch.stack([(packed >> s) & 3 for s in (0, 2, 4, 6)], 1).view(-1)
    regs = torch.zeros(dbg.SKETCH_REGISTERS, dtype=torch.int64, device=DEV)
    lens = offsets.diff()
    for r0 in range(0, lens.numel(), 1 << 18):
        r1 = min(lens.numel(), r0 + (1 << 18))
        b0, b1 = int(offsets[r0]), int(offsets[r1])
        c = codes[b0:b1].long()
        if c.numel() < m:
            continue
        keys = torch.zeros(c.numel() - m + 1, dtype=torch.int64, device=DEV)
        for j in range(m):
            keys = (keys << 2) | c[j:j + keys.numel()]
        end = torch.repeat_interleave(offsets[r0 + 1:r1 + 1] - b0, lens[r0:r1],
                                      output_size=b1 - b0)
        size = torch.repeat_interleave(lens[r0:r1], lens[r0:r1], output_size=b1 - b0)
        at = torch.arange(keys.numel(), device=DEV)
        x = keys[(at + m <= end[:keys.numel()]) & (size[:keys.numel()] >= k)] ^ _SALT
        x = (x ^ _shift(x, 33)) * _M1
        x = (x ^ _shift(x, 33)) * _M2
        x = x ^ _shift(x, 33)
        rest = x & ((1 << 54) - 1)  # its leading zeros among 54 bits, by halving
        rho = torch.ones_like(rest)
        width = 54
        for step in (27, 14, 7, 4, 2, 1):
            low = _shift(rest, width - step) == 0 if width > step else rest == 0
            rho += torch.where(low, min(step, width), 0)
            rest = torch.where(low, rest << min(step, width), rest) & ((1 << 54) - 1)
        regs.scatter_reduce_(0, _shift(x, 54), rho.clamp(max=55), "amax")
    return regs


def exact(case, seed):
    if case["do"] not in ("size", "train"):
        return None
    s = prepare(case, seed)
    if case["do"] == "size":
        regs = torch.stack([_registers(k, p, o) for k, p, o, _ in s["items"]])
        return _forward(s["params"].double(), regs.double() / 64), None
    b, t = case["batch"], s["step"] + 1
    p = s["params"].double().requires_grad_(True)
    loss = 0.5 * (_forward(p, s["x"].double()) - s["target"].double()).square().sum() / b
    (g,) = torch.autograd.grad(loss, p)
    m = 0.9 * s["m"].double() + 0.1 * g
    v = 0.999 * s["v"].double() + 0.001 * g * g
    new = p.detach() - 1e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return {"params": new, "grads": g, "m": m, "v": v, "loss": loss.detach().view(1)}

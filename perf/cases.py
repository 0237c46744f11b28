"""What a user of the engine has it do, as cases that can be timed and compared.

A case is one call sequence of a training program: score every neighbourhood ("eval"), train
some iterations and read the state back ("train"), the same with minibatches from the host
("stream"), one step whose gradients are read back ("grads"), and the fitness of logits that are
already on the device ("fitness"). Sizes are those of the repository's configurations, tests and
benchmark: 1x1 to 12x12 tori, fp32 and bf16, the MLP and DCGAN networks of Table 1, batch 100, 128
and 256, and widths that fill no tile.

Results are read into pinned host memory, as a program that cares for speed does. The state of a
training case comes back whole (weights, both moments, step counts, learning rates, mixture
weights) through lipz_export_state, as at a checkpoint.
"""

import math

import torch

import paper_1811_12843_gb300 as L

FP64 = torch.float64

_DEFAULTS = dict(rows=1, cols=1, precision="bf16", batch=100, net="mlp", z=64, hidden=256,
                 x=784, width=64, iters=1, steps=1, mixture=False, stale=False, pool=8192)


def _case(name, op, **kw):
    c = dict(_DEFAULTS, op=op, **kw)
    if name:
        c["name"] = name
    return c


def _dcgan(**kw):
    return dict(net="dcgan", z=100, x=12288, pool=2000, **kw)


def listed():
    return [
        # a serving loop that has the logits on the device and wants the fitness: the smallest call
        _case("fitness_2x2", "fitness", rows=2, cols=2),
        # the smallest grid of the configurations, in fp32: scoring alone
        _case("eval_2x2_fp32", "eval", rows=2, cols=2, precision="fp32"),
        # the 3x3 fp32 configuration: twenty iterations, then a checkpoint
        _case("train_3x3_fp32_x20", "train", rows=3, cols=3, precision="fp32", iters=20),
        # sizes that fill no tile, in bf16 (CUDA-core kernels), one step with its gradients
        _case("grads_3x4_ragged", "grads", rows=3, cols=4, batch=37, z=50, hidden=200, x=500),
        # the 1x1 grid (one GAN, the baseline of the grid comparisons): latency of one cell
        _case("train_1x1_bf16_x20", "train", iters=20),
        # the 5x5 batch-256 configuration: scoring with the mixture step, and ten iterations
        _case("eval_5x5_bf16_b256_mix", "eval", rows=5, cols=5, batch=256, mixture=True),
        _case("train_5x5_bf16_b256_x10", "train", rows=5, cols=5, batch=256, iters=10),
        # an 8x8 grid fed by a host data loader, pipelined one call ahead
        _case("stream_8x8_bf16_x4", "stream", rows=8, cols=8, iters=4),
        # the benchmark's grid: scoring alone, and training with a checkpoint at the end
        _case("eval_12x12_bf16", "eval", rows=12, cols=12, pool=60000),
        _case("train_12x12_bf16_x4", "train", rows=12, cols=12, iters=4, pool=60000),
        # the 3x3 DCGAN configuration: scoring alone, and two iterations
        _case("eval_3x3_dcgan", "eval", rows=3, cols=3, batch=128, **_dcgan()),
        _case("train_3x3_dcgan_x2", "train", rows=3, cols=3, batch=128, iters=2, **_dcgan()),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more call of the same kinds: grids, batches and options over the ranges above."""
    op = rng.choice(["fitness", "eval", "eval", "train", "train", "train", "stream", "grads"])
    if op == "fitness":
        cells = _log(rng, 1, 144)
        return _case(None, op, rows=1, cols=cells, batch=_log(rng, 16, 256))
    if op == "grads":
        return _case(None, op, rows=rng.randint(1, 4), cols=rng.randint(1, 5),
                     precision=rng.choice(["fp32", "bf16"]), batch=_log(rng, 8, 128),
                     z=rng.randint(16, 100), hidden=rng.choice([64, 200, 256, 300, 512]),
                     x=rng.choice([64, 500, 784, 1000]))
    if op != "stream" and rng.random() < 0.25:
        return _case(None, op, rows=rng.randint(1, 3), cols=rng.randint(1, 3),
                     batch=_log(rng, 16, 112), iters=rng.randint(1, 2) if op == "train" else 1,
                     **_dcgan())
    fp32 = op != "stream" and rng.random() < 0.35
    side = 4 if fp32 else 12
    rows, cols = _log(rng, 1, side), _log(rng, 1, side)
    batch = _log(rng, 16, 256)
    while rows * cols * batch > (1600 if fp32 else 14400):
        batch = max(16, batch // 2)
    kw = dict(rows=rows, cols=cols, batch=batch, precision="fp32" if fp32 else "bf16")
    if op == "eval":
        kw["mixture"] = rng.random() < 0.3
    else:
        kw["iters"] = rng.randint(2, max(3, min(12, 600 // (rows * cols))))
        if op == "train" and rng.random() < 0.25:
            kw["steps"] = rng.randint(2, 3)
        elif op == "train" and rng.random() < 0.25:
            kw["stale"] = True
    return _case(None, op, **kw)


# ---- inputs -----------------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _blobs(seed, n, dim):
    """n rows in [-1, 1] around ten blob centres (what stands in for MNIST), on the GPU."""
    g = _gen(seed)
    centres = torch.rand((10, dim), generator=g, device="cuda") * 2 - 1
    which = torch.randint(0, 10, (n,), generator=g, device="cuda")
    noise = torch.randn((n, dim), generator=g, device="cuda")
    return (centres[which] + 0.3 * noise).clamp_(-1, 1)


def _fields(seed, n):
    """n smooth 3x64x64 random fields in [-1, 1] (what stands in for CelebA), on the GPU."""
    g = _gen(seed)
    f = torch.fft.fftfreq(64, device="cuda")
    filt = torch.exp(-2.0 * (math.pi * 4.0) ** 2 * (f[:, None] ** 2 + f[None, :] ** 2))
    out = []
    for s in range(0, n, 500):
        w = torch.randn((min(500, n - s), 3, 64, 64), generator=g, device="cuda")
        sm = torch.fft.ifft2(torch.fft.fft2(w) * filt).real
        out.append((sm / sm.abs().amax(dim=(2, 3), keepdim=True)).reshape(-1, 12288))
    return torch.cat(out)


def _pool(case, seed):
    return (_fields(seed, case["pool"]) if case["net"] == "dcgan"
            else _blobs(seed, case["pool"], case["x"]))


def _logits(case, seed):
    """Logits as a discriminator in training gives them, [cells][5][6 batch]."""
    c = case["rows"] * case["cols"]
    return 2.0 * torch.randn((c, 5, 6 * case["batch"]), generator=_gen(seed), device="cuda")


def _pinned(*shape, dtype=torch.float32):
    return torch.empty(shape, dtype=dtype, pin_memory=True)


def _counts(case):
    return L.param_counts(case["z"], case["hidden"], case["x"],
                          L.LIPZ_DCGAN64 if case["net"] == "dcgan" else L.LIPZ_MLP,
                          case["width"], case["width"])


def prepare(case, seed):
    C, B = case["rows"] * case["cols"], case["batch"]
    if case["op"] == "fitness":
        return {"case": case, "logits": _logits(case, seed),
                "fit_g": torch.zeros((C, 5), device="cuda"),
                "fit_d": torch.zeros((C, 5), device="cuda"),
                "stream": torch.cuda.current_stream().cuda_stream}
    kw = dict(precision=case["precision"], batch=B, z_dim=case["z"], x_dim=case["x"],
              train_steps=case["steps"], mixture=int(case["mixture"]),
              stale_neighbors=int(case["stale"]))
    if case["net"] == "dcgan":
        kw.update(kind=L.LIPZ_DCGAN64, ngf=case["width"], ndf=case["width"], lr=5e-5)
    else:
        kw.update(hidden=case["hidden"])
    if case["op"] == "grads":
        # every centre is replaced by a random neighbour: the step does not hang on fitness ties
        kw.update(keep_grads=1, tournament_size=1, replace_mode="always")
    g = L.Grid(case["rows"], case["cols"], seed=seed, **kw)
    s = {"case": case, "grid": g, "fit_g": _pinned(C, 5), "fit_d": _pinned(C, 5)}
    pool = _pool(case, seed)
    if case["op"] == "stream":
        # the loader's minibatches, pinned, and one pair of result buffers for each call
        pick = torch.randint(0, case["pool"], (case["iters"], C * B), generator=_gen(seed + 1),
                             device="cuda")
        s["x"] = [pool[p].reshape(C, B, case["x"]).cpu().pin_memory() for p in pick]
        s["fits"] = [(_pinned(C, 5), _pinned(C, 5)) for _ in range(case["iters"])]
    else:
        g.set_data(pool.cpu().numpy())
    if case["op"] == "eval":
        s["pair_g"], s["pair_d"] = _pinned(C, 5, 5), _pinned(C, 5, 5)
        s["logits"] = _pinned(C, 5, 6 * B)
        if case["mixture"]:
            s["mix"] = (_pinned(C, 5), _pinned(C, 6, 6), _pinned(C))
    elif case["op"] == "grads":
        s["grad_g"], s["grad_d"] = _pinned(C, g.PG), _pinned(C, g.PD)
    if case["op"] in ("train", "stream"):
        s["state"] = _pinned(L.lipz_state_bytes(g.h), dtype=torch.uint8)
    return s


def _checkpoint(s):
    """The grid's state in the caller's pinned buffer, as its named parts (views)."""
    g, buf = s["grid"], s["state"]
    rc = L.load().lipz_export_state(g.h, buf.data_ptr(), buf.numel())
    if rc:
        raise L.LipzError(rc, L.lipz_last_error(g.h))
    C, off, out = g.cells, 64, {}
    for name, shape, kind in [("Gw", (C, g.PG), torch.float32), ("Gm", (C, g.PG), torch.float32),
                              ("Gv", (C, g.PG), torch.float32), ("Dw", (C, g.PD), torch.float32),
                              ("Dm", (C, g.PD), torch.float32), ("Dv", (C, g.PD), torch.float32),
                              ("Gstep", (C,), torch.int32), ("Dstep", (C,), torch.int32),
                              ("Glr", (C,), torch.float32), ("Dlr", (C,), torch.float32),
                              ("mix", (C, 5), torch.float32)]:
        n = 4 * math.prod(shape)
        out[name] = buf[off:off + n].view(kind).reshape(shape)
        off += n
    return out


def run(state):
    s, case = state, state["case"]
    op = case["op"]
    if op == "fitness":
        L.lipz_fitness_from_logits_noalloc(s["logits"], case["rows"] * case["cols"],
                                           case["batch"], s["fit_g"], s["fit_d"], s["stream"])
        return {"fit_g": s["fit_g"], "fit_d": s["fit_d"]}
    h = s["grid"].h
    if op == "eval":
        L.lipz_eval_neighborhoods(h, s["fit_g"], s["fit_d"], s["pair_g"], s["pair_d"])
        L.lipz_get_logits(h, s["logits"])
        out = {k: s[k] for k in ("fit_g", "fit_d", "pair_g", "pair_d", "logits")}
        if case["mixture"]:
            L.lipz_get_mixture(h, *s["mix"])
            out.update(zip(("mix_w", "mix_blocks", "mix_score"), s["mix"]))
        return out
    if op == "train":
        L.lipz_iterate(h, case["iters"])
        return _checkpoint(s)
    if op == "stream":
        xs, n = s["x"], case["iters"]
        for i in range(n):
            L.lipz_iterate_batch_async(h, xs[i], xs[i + 1] if i + 1 < n else None, *s["fits"][i])
        L.lipz_synchronize(h)
        return dict(_checkpoint(s), fits=s["fits"])
    L.lipz_eval_neighborhoods(h, s["fit_g"], s["fit_d"])
    L.lipz_select_replace(h)
    L.lipz_train_step(h)
    L.lipz_get_gradients(h, s["grad_g"], s["grad_d"])
    return {k: s[k] for k in ("fit_g", "fit_d", "grad_g", "grad_d")}


# ---- what a pass cannot do without ------------------------------------------------------------
def _macs(case):
    """Multiply-adds of one sample's forward: (generator, generator without its output layer,
    discriminator)."""
    if case["net"] == "dcgan":
        w, z = case["width"], case["z"]
        g = z * 8 * w * 16 + 16 * 8 * w * 4 * w * 16 + 64 * 4 * w * 2 * w * 16 \
            + 256 * 2 * w * w * 16
        out = 1024 * w * 3 * 16
        d = 1024 * w * 3 * 16 + 256 * 2 * w * w * 16 + 64 * 4 * w * 2 * w * 16 \
            + 16 * 8 * w * 4 * w * 16 + 8 * w * 16
        return g + out, g, d
    z, h, x = case["z"], case["hidden"], case["x"]
    return z * h + h * h + h * x, z * h + h * h, x * h + h * h + h


def work(case):
    C, B, x = case["rows"] * case["cols"], case["batch"], case["x"]
    if case["op"] == "fitness":
        return {"bytes": C * (30 * B + 10) * 4, "flops": C * 55 * B * 4}
    bf = case["precision"] == "bf16"
    es = 2 if bf else 4
    PG, PD = _counts(case)
    g, g_hid, d = _macs(case)
    # scoring: 5 generators on B rows, 5 discriminators on 6 B rows of every cell; every
    # individual's weights and every real row read once, the logits written
    ev_flops = 2 * C * (5 * B * g + 30 * B * d)
    ev_bytes = C * ((PG + PD) * es + B * x * es + 30 * B * 4)
    if case["mixture"]:
        ev_flops += 2 * C * (6 * B) ** 2 * x
    if case["op"] == "eval":
        return {"bytes": ev_bytes + C * 30 * B * 4, "flops": ev_flops}
    # a training step: the pair's forward (2 B rows through D) and backward (weight gradients of
    # both; deltas through D for 3 B rows and through G)
    tr_flops = 2 * C * B * (g_hid + 2 * d + 2 * d + 3 * d + 2 * g)
    # Adam: w, m, v read and written, and the bf16 copy written
    tr_bytes = C * (PG + PD) * (26 if bf else 24)
    if case["op"] == "grads":
        return {"bytes": ev_bytes + tr_bytes + C * (PG + PD) * 8, "flops": ev_flops + tr_flops}
    n, k = case["iters"], case["steps"]
    more = 2 * C * B * g * (k - 1)
    total = n * (ev_bytes + k * tr_bytes) + C * (PG + PD) * 24
    if case["op"] == "stream":
        total += n * C * B * x * 4
    return {"bytes": total, "flops": n * (ev_flops + k * tr_flops + more)}


def tolerance(case):
    """Measured. fp32: against 64 bits. bf16: against the same call with the start's weights moved
    by 1e-7 (relative), which moves some values over a bf16 rounding boundary as another order of
    the sums would: the moments of MLP training then differ by up to 1.2e-2 (fewer than nine
    iterations; later a tournament goes the other way), those of DCGAN training by 2.6e-2."""
    op, fp32 = case["op"], case["precision"] == "fp32"
    if op == "fitness":
        return {"rel": 1e-6}
    if op == "eval":
        return {"rel": 1e-5 if fp32 else 2e-2 if case["net"] == "dcgan" else 1e-2}
    if op == "grads":
        return {"rel": 1e-3 if fp32 else 2e-2, "max": 1e-1 if fp32 else 0.9}
    return {"rel": 4e-3 if fp32 and case["net"] == "mlp" else 3e-2, "max": 0.99}


# ---- the same in 64 bits ----------------------------------------------------------------------
def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors of 32-bit words: the four output words, stacked last."""
    m = 0xFFFFFFFF
    c0, c1, c2, c3 = torch.broadcast_tensors(*(torch.as_tensor(v, device="cuda")
                                               for v in (c0, c1, c2, c3)))

    def mul(a, c):
        # the 64-bit product's halves; the upper one from 16-bit pieces of the constant
        return ((a >> 16) * c + ((a & 0xFFFF) * c >> 16)) >> 16, (a * c) & m

    k0, k1 = seed & m, seed >> 32 & m
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
    return torch.stack([c0, c1, c2, c3], -1)


def _words(seed, stream, t, C, n):
    """The first n words of (stream, t, cell) for every cell, [C, n]."""
    blk = torch.arange((n + 3) // 4, device="cuda")[None]
    cell = torch.arange(C, device="cuda")[:, None]
    return _philox(blk, cell, t, stream, seed).reshape(C, -1)[:, :n]


def _normals(seed, stream, t, C, n):
    w = _words(seed, stream, t, C, (n + 3) // 4 * 4).reshape(C, -1, 2)
    r = torch.sqrt(-2 * torch.log(((w[..., 0] >> 8) + 1).to(FP64) * 2.0 ** -24))
    a = 2 * math.pi * ((w[..., 1] >> 8).to(FP64) * 2.0 ** -24)
    return torch.stack([r * torch.cos(a), r * torch.sin(a)], -1).reshape(C, -1)[:, :n]


def _shapes(case):
    """The parameter tensors of a generator and a discriminator, in storage order."""
    if case["net"] == "dcgan":
        w = case["width"]
        ch, dh = [case["z"], 8 * w, 4 * w, 2 * w, w], [3, w, 2 * w, 4 * w, 8 * w]
        g = []
        for i in range(4):
            g += [(ch[i], ch[i + 1], 4, 4), (ch[i + 1],), (ch[i + 1],)]
        return g + [(w, 3, 4, 4)], [(dh[i + 1], dh[i], 4, 4) for i in range(4)] + [(1, 8 * w, 4, 4)]
    z, h, x = case["z"], case["hidden"], case["x"]
    return [(h, z), (h,), (h, h), (h,), (x, h), (x,)], [(h, x), (h,), (h, h), (h,), (1, h), (1,)]


def _split(flat, shapes):
    out, off = [], 0
    for s in shapes:
        n = math.prod(s)
        out.append(flat[..., off:off + n].reshape(flat.shape[:-1] + s))
        off += n
    return out


def _init(case, seed, stream, shapes):
    C = case["rows"] * case["cols"]
    n = sum(math.prod(s) for s in shapes)
    if case["net"] == "dcgan":
        # weights N(0, 0.02^2), batch-norm scales 1 + N(0, 0.02^2), shifts 0
        p = (0.02 * _normals(seed, stream, 0, C, n))
        off = 0
        for k, s in enumerate(shapes):
            m = math.prod(s)
            if len(s) == 1:
                p[:, off:off + m] = 1 + p[:, off:off + m] if k % 3 == 1 else 0.0
            off += m
    else:
        # Xavier-uniform weights, zero biases
        q = (2 * (_words(seed, stream, 0, C, n) >> 8) + 1 - 2 ** 24).to(FP64) * 2.0 ** -24
        off, p = 0, torch.zeros_like(q)
        for k, s in enumerate(shapes):
            m = math.prod(s)
            if k % 2 == 0:
                a = torch.tensor(math.sqrt(6.0 / (s[0] + s[1])), dtype=torch.float32).item()
                p[:, off:off + m] = a * q[:, off:off + m]
            off += m
    return p.float().to(FP64)


def _neighbours(case):
    R, Q = case["rows"], case["cols"]
    c = torch.arange(R * Q, device="cuda")
    r, q = c // Q, c % Q
    return torch.stack([c, (r - 1) % R * Q + q, (r + 1) % R * Q + q, r * Q + (q - 1) % Q,
                        r * Q + (q + 1) % Q], 1)


def _conv(x, w, s, p):
    n, _, h, _ = x.shape
    u = torch.nn.functional.unfold(x, 4, padding=p, stride=s)
    o = (h + 2 * p - 4) // s + 1
    return (w.reshape(w.shape[0], -1) @ u).reshape(n, w.shape[0], o, o)


def _convt(x, w, s, p):
    n, c, h, _ = x.shape
    u = w.reshape(c, -1).T @ x.reshape(n, c, h * h)
    o = s * (h - 1) + 4 - 2 * p
    return torch.nn.functional.fold(u, o, 4, padding=p, stride=s)


def _lrelu(v):
    return torch.where(v > 0, v, torch.tensor(0.2, dtype=torch.float32).item() * v)


def _generator(case, W, z):
    """Fakes [C, B, x] of the C generators W on z [C, B, z]."""
    if case["net"] == "dcgan":
        out = []
        for c in range(z.shape[0]):
            v = z[c][:, :, None, None]
            for i in range(4):
                v = _convt(v, W[3 * i][c], 1 if i == 0 else 2, 0 if i == 0 else 1)
                mean = v.mean((0, 2, 3), keepdim=True)
                var = ((v - mean) ** 2).mean((0, 2, 3), keepdim=True)
                v = (v - mean) / torch.sqrt(var + 1e-5) * W[3 * i + 1][c][:, None, None] \
                    + W[3 * i + 2][c][:, None, None]
                v = v.clamp(min=0)
            out.append(torch.tanh(_convt(v, W[12][c], 2, 1)).reshape(z.shape[1], -1))
        return torch.stack(out)
    h = (z @ W[0].mT + W[1][:, None]).clamp(min=0)
    h = (h @ W[2].mT + W[3][:, None]).clamp(min=0)
    return torch.tanh(h @ W[4].mT + W[5][:, None])


def _discriminator(case, W, X):
    """Logits [C, rows] of the C discriminators W on X [C, rows, x]."""
    if case["net"] == "dcgan":
        out = []
        for c in range(X.shape[0]):
            rows = []
            for part in X[c].split(128):
                v = part.reshape(-1, 3, 64, 64)
                for i in range(4):
                    v = _lrelu(_conv(v, W[i][c], 2, 1))
                rows.append(v.reshape(v.shape[0], -1) @ W[4][c].reshape(-1))
            out.append(torch.cat(rows))
        return torch.stack(out)
    h = _lrelu(X @ W[0].mT + W[1][:, None])
    h = _lrelu(h @ W[2].mT + W[3][:, None])
    return (h @ W[4].mT + W[5][:, None])[..., 0]


def _fitness(logits, B):
    sp = torch.nn.functional.softplus
    C = logits.shape[0]
    l = logits.reshape(C, 5, 6, B)  # [c][j][real, fakes of slot i][b]
    real = sp(-l[:, :, 0]).mean(-1)
    lg = sp(-l[:, :, 1:]).mean(-1).mT  # [c][i][j]
    ld = real[:, None] + sp(l[:, :, 1:]).mean(-1).mT
    return {"fit_g": lg.mean(2), "fit_d": ld.mean(1), "pair_g": lg, "pair_d": ld}


def _minibatch(case, seed, t, pool):
    C, B = case["rows"] * case["cols"], case["batch"]
    idx = _words(seed, 3, t, C, B) * pool.shape[0] >> 32
    return pool[idx].to(FP64), _normals(seed, 4, t, C, B * case["z"]).reshape(C, B, -1)


def _score(case, Gs, Ds, shapes, x, z):
    nbr = _neighbours(case)
    X = torch.cat([x] + [_generator(case, _split(Gs[nbr[:, i]], shapes[0]), z)
                         for i in range(5)], 1)
    logits = torch.stack([_discriminator(case, _split(Ds[nbr[:, j]], shapes[1]), X)
                          for j in range(5)], 1)
    return X, dict(_fitness(logits, case["batch"]), logits=logits)


def _select(seed, stream, t, fit, size, always):
    C = fit.shape[0]
    w, f = _words(seed, stream, t, C, 5).tolist(), fit.tolist()
    sel = []
    for c in range(C):
        left = [0, 1, 2, 3, 4]
        got = [left.pop(w[c][m] * (5 - m) >> 32) for m in range(size)]
        win = min(got, key=lambda e: (f[c][e], e))
        sel.append(win if always or f[c][win] < f[c][0] else 0)
    return torch.tensor(sel, device="cuda")


def _gradients(case, Gs, Ds, shapes, x, z):
    """dL_G / dG and dL_D / dD of every cell's pair, by autograd in 64 bits."""
    sp = torch.nn.functional.softplus
    with torch.enable_grad():
        G, D = Gs.clone().requires_grad_(True), Ds.clone().requires_grad_(True)
        fakes = _generator(case, _split(G, shapes[0]), z)
        W = _split(D, shapes[1])
        l_g = sp(-_discriminator(case, W, fakes)).mean(1).sum()
        l_d = (sp(-_discriminator(case, W, x)).mean(1)
               + sp(_discriminator(case, W, fakes.detach())).mean(1)).sum()
        return torch.autograd.grad(l_g, G)[0], torch.autograd.grad(l_d, D)[0]


@torch.no_grad()
def exact(case, seed):
    """Plain 64-bit torch. None for bf16 training over several iterations: tournaments and Adam's
    first steps, which move an element by the sign of its gradient, carry bf16 rounding on from
    one iteration to the next, and 64 bits would follow another path."""
    op, B = case["op"], case["batch"]
    if op == "fitness":
        f = _fitness(_logits(case, seed).to(FP64), B)
        return {"fit_g": f["fit_g"], "fit_d": f["fit_d"]}
    fp32 = case["precision"] == "fp32"
    if op == "stream" or (op == "train" and not (fp32 and case["steps"] == 1
                                                 and not case["stale"])):
        return None
    shapes = _shapes(case)
    C = case["rows"] * case["cols"]
    G, D = (_init(case, seed, 1 + k, shapes[k]) for k in range(2))
    pool = _pool(case, seed)
    nbr = _neighbours(case)
    if op == "eval":
        x, z = _minibatch(case, seed, 0, pool)
        X, out = _score(case, G, D, shapes, x, z)
        if case["mixture"]:
            n2 = (X * X).sum(-1)
            S = torch.exp(-(n2[:, :, None] + n2[:, None] - 2 * X @ X.mT) / case["x"])
            out.update(mix_w=None, mix_score=None,
                       mix_blocks=S.reshape(C, 6, B, 6, B).mean((2, 4)))
        return out
    lr, b1, b2, eps = (torch.tensor(v, dtype=torch.float32).item()
                       for v in (2e-4, 0.5, 0.999, 1e-8))
    pops = [dict(w=w, m=torch.zeros_like(w), v=torch.zeros_like(w),
                 step=torch.zeros(C, dtype=torch.int64, device="cuda")) for w in (G, D)]
    for t in range(case["iters"]):
        x, z = _minibatch(case, seed, t, pool)
        fit = _score(case, pops[0]["w"], pops[1]["w"], shapes, x, z)[1]
        new = []
        for k, f in enumerate(("fit_g", "fit_d")):
            sel = _select(seed, 5 + k, t, fit[f], 1 if op == "grads" else 2, op == "grads")
            src = nbr[torch.arange(C, device="cuda"), sel]
            new.append({n: v[src] for n, v in pops[k].items()})
        grads = _gradients(case, new[0]["w"], new[1]["w"], shapes, x, z)
        if op == "grads":
            return {"fit_g": fit["fit_g"], "fit_d": fit["fit_d"], "grad_g": grads[0],
                    "grad_d": grads[1]}
        for p, g in zip(new, grads):
            p["step"] = p["step"] + 1
            n = p["step"].to(FP64)[:, None]
            p["m"] = b1 * p["m"] + (1 - b1) * g
            p["v"] = b2 * p["v"] + (1 - b2) * g * g
            p["w"] = p["w"] - lr * (p["m"] / (1 - b1 ** n)) / (
                torch.sqrt(p["v"] / (1 - b2 ** n)) + eps)
        pops = new
    out = {k + n: p[n] for k, p in zip("GD", pops) for n in ("w", "m", "v")}
    rates = torch.full((C,), lr, dtype=FP64, device="cuda")
    return dict(out, Glr=rates, Dlr=rates, mix=torch.full((C, 5), 0.2, dtype=FP64, device="cuda"))

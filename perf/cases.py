"""Workloads for timing the library: block-sparse products and the cost model's training.

A case names a block structure (a recipe of ``bsmm_gen`` with its sizes and a pattern
number that fixes tilings and masks), a precision mode and the plan's options. The values
are drawn on the GPU from the seed. ``run`` is one call of the public entry point a program
makes: ``bsmm_execute`` (``bsmm_execute_f32``), ``bsmm_batch_execute``,
``bsmm_split_tile_noalloc`` or the training calls of ``costmodel.fit``.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import bsmm_gen as G
import paper_1504_05046_gb300 as P

MODES = {"fp64": P.BSMM_FP64, "bf16": P.BSMM_SPLIT_BF16, "fp16": P.BSMM_SPLIT_FP16}
ELEMS = {"f64": (P.BSMM_F64, torch.float64, 2), "f32": (P.BSMM_F32, torch.float32, 4),
         "c128": (P.BSMM_C128, torch.complex128, 2)}


def _product(name, recipe, n, mode, **kw):
    c = {"name": name, "kind": "product", "recipe": recipe, "n": n, "mode": mode, "s": 6, "elem": "f64", "lo": 64,
         "hi": 256, "density": 0.5, "band": 6, "k_factor": 2, "pattern": 1, "alpha": 1.0, "beta": 0.0, "transa": 0,
         "transb": 0, "split_scale": 0, "cluster": -1, "ksplit": 0}
    c.update(kw)
    return c


def listed():
    return [
        # one dense tile task of odd sizes without any allocation: the smallest call, all latency
        {"name": "tile 200x136x311", "kind": "tile", "m": 200, "n": 136, "k": 311, "s": 6, "alpha": -0.5, "beta": 0.5},
        # a small dense product of ragged tiles (launches and latency count), C accumulated
        _product("split small 1100", "nonuniform_dense", 1100, "bf16", beta=0.5, cluster=0),
        # the paper's uniform square workload with random tile masks, split and plain FP64
        _product("split uniform 2048", "uniform_bernoulli", 2048, "bf16"),
        _product("fp64 uniform 2048", "uniform_bernoulli", 2048, "fp64", cluster=0),
        # the paper's nonuniform square workload at half its size (N = 32768): the headline
        _product("split dense 16384", "nonuniform_dense", 16384, "bf16"),
        # banded operators with distance decay (electronic-structure matrices), float16 slices
        _product("split banded 32768", "banded_decay", 32768, "fp16", lo=32, hi=256),
        # irregular clusters of nonzero tiles, tile sizes from 16 to 512, rectangular
        _product("split clustered 24576", "clustered", 24576, "bf16", lo=16, hi=512, density=0.10),
        # few C tiles and a very long inner dimension (contraction of tall operands): split k
        _product("split thin 512x524288", "thin_dense", 512, "bf16", k_factor=1024),
        # single precision data with 4 slices
        _product("f32 dense 8192", "nonuniform_dense", 8192, "bf16", s=4, elem="f32"),
        # complex data, A stored transposed, one scale per row and column
        _product("complex dense 3072", "nonuniform_dense", 3072, "bf16", elem="c128", transa=1, split_scale=1),
        # many independent products of uneven sizes and densities in one call
        {"name": "batch 48", "kind": "batch", "count": 48, "n_lo": 512, "n_hi": 4096, "b_lo": 32, "b_hi": 192,
         "d_lo": 0.1, "d_hi": 1.0, "mode": "bf16", "s": 6, "pattern": 1},
        # training the task-cost model on the unit times of a few products, and predicting with it
        {"name": "cost model fit", "kind": "fit", "rows": 20000, "steps": 300, "lr": 3e-3},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tile", "dense", "dense", "uniform", "banded", "banded", "clustered", "thin", "batch", "fp64",
                       "fp64", "fit"])
    pat = rng.randrange(2, 1000)
    if kind == "tile":
        return {"kind": "tile", "m": rng.randint(1, 256), "n": rng.randint(1, 256), "k": rng.randint(1, 512),
                "s": rng.randint(3, 6), "alpha": rng.choice([1.0, -0.5]), "beta": rng.choice([0.0, 0.5])}
    if kind == "fit":
        return {"kind": "fit", "rows": _log(rng, 300, 40000), "steps": _log(rng, 20, 400), "lr": 3e-3}
    if kind == "batch":
        hi = _log(rng, 700, 4096)
        return {"kind": "batch", "count": rng.randint(2, 48), "n_lo": min(512, hi), "n_hi": hi, "b_lo": 32,
                "b_hi": rng.randint(64, 192), "d_lo": 0.1, "d_hi": 1.0, "mode": rng.choice(["bf16", "fp16", "fp64"])
                if hi <= 1500 else rng.choice(["bf16", "fp16"]), "s": rng.choice([4, 6, 6]), "pattern": pat}
    opt = {"pattern": pat, "alpha": rng.choice([1.0, 1.0, -0.5]), "beta": rng.choice([0.0, 0.0, 0.5]),
           "transa": rng.choice([0, 0, 1]), "transb": rng.choice([0, 0, 1])}
    if kind == "fp64":
        recipe = rng.choice(["uniform_bernoulli", "nonuniform_dense", "banded_decay", "clustered"])
        n = _log(rng, *{"uniform_bernoulli": (200, 4096), "nonuniform_dense": (200, 3000),
                        "banded_decay": (600, 12000), "clustered": (4000, 7000)}[recipe])
        c = _product("", recipe, n, "fp64", cluster=0, density=0.10 if recipe == "clustered" else 0.5,
                     lo=16 if recipe == "clustered" else 32, hi=512 if recipe == "clustered" else 256, **opt)
    else:
        opt.update(s=rng.choice([3, 4, 6, 6, 6]), elem=rng.choice(["f64", "f64", "f32", "c128"]),
                   split_scale=rng.choice([0, 0, 1]), cluster=rng.choice([-1, -1, 0]))
        mode = rng.choice(["bf16", "bf16", "fp16"])
        if opt["elem"] == "f32":
            opt["alpha"] = float(np.float32(opt["alpha"]))
        if kind == "dense":
            c = _product("", "nonuniform_dense", _log(rng, 300, 8192), mode, **opt)
        elif kind == "uniform":
            c = _product("", "uniform_bernoulli", _log(rng, 300, 8192), mode, density=rng.uniform(0.2, 0.9), **opt)
        elif kind == "banded":
            c = _product("", "banded_decay", _log(rng, 1000, 32768), mode, lo=32, hi=256, band=rng.randint(2, 8), **opt)
        elif kind == "clustered":
            c = _product("", "clustered", _log(rng, 4000, 16000), mode, lo=16, hi=512, density=0.10, **opt)
        else:
            c = _product("", "thin_dense", rng.randint(100, 600), mode, k_factor=_log(rng, 64, 512), **opt)
    del c["name"]
    return c


# ---------------------------------------------------------------- block structures
class _Structure:
    """Tilings, masks and arena layouts of one product (host arrays, no values)."""

    def __init__(self, r, c, q, am, bm, transa=0, transb=0, align=2):
        self.r, self.c, self.q, self.am, self.bm = r, c, q, am, bm  # masks in (i,k) and (k,j)
        self.transa, self.transb = transa, transb
        self.a_mask = np.ascontiguousarray(am.T) if transa else am
        self.b_mask = np.ascontiguousarray(bm.T) if transb else bm
        self.a_off, self.a_len = G.layout_arena(self.a_mask, *((q, r) if transa else (r, q)), align=align)
        self.b_off, self.b_len = G.layout_arena(self.b_mask, *((c, q) if transb else (q, c)), align=align)
        self.cs = (am.astype(np.int64) @ bm.astype(np.int64) > 0).astype(np.uint8)
        self.c_off, self.c_len = G.layout_arena(self.cs, r, c, align=align)

    def useful_flops(self):
        return 2.0 * float(np.einsum("i,ik,k,kj,j->", self.r.astype(float), self.am.astype(float),
                                     self.q.astype(float), self.bm.astype(float), self.c.astype(float),
                                     optimize=True))

    def elements(self):
        stored = [float(x.astype(float) @ m.astype(float) @ y.astype(float))
                  for x, m, y in ((self.r, self.am, self.q), (self.q, self.bm, self.c), (self.r, self.cs, self.c))]
        return stored


def _streams(pattern):
    return [np.random.default_rng(s) for s in np.random.SeedSequence(pattern).spawn(2)]


def _structure(case):
    rt, rm = _streams(case["pattern"])
    n, lo, hi, recipe = case["n"], case["lo"], case["hi"], case["recipe"]
    if recipe == "uniform_bernoulli":
        r = c = q = G.tiling_uniform(n, 128)
        am, bm = (G.mask_bernoulli(len(r), len(r), case["density"], rm) for _ in range(2))
    elif recipe == "nonuniform_dense":
        r = c = q = G.tiling_uniform_int(n, lo, hi, rt)
        am = bm = G.mask_dense(len(r), len(r))
    elif recipe == "banded_decay":
        r = c = q = G.tiling_uniform_int(n, lo, hi, rt)
        am = bm = G.mask_band(len(r), len(r), case["band"])
    elif recipe == "clustered":
        r, c, q = (G.tiling_log_uniform(m, lo, hi, rt) for m in (n, n, case["k_factor"] * n))
        clusters = 40 if n >= 12000 else 12  # fewer on the coarser tile grids of smaller matrices
        am = G.mask_clusters(len(r), len(q), clusters, case["density"], rm, tol=0.03)
        bm = G.mask_clusters(len(q), len(c), clusters, case["density"], rm, tol=0.03)
    elif recipe == "thin_dense":
        r = c = G.tiling_uniform_int(n, lo, hi, rt)
        q = G.tiling_uniform_int(case["k_factor"] * n, lo, hi, rt)
        am, bm = G.mask_dense(len(r), len(q)), G.mask_dense(len(q), len(c))
    else:
        raise ValueError(recipe)
    return _Structure(r, c, q, am, bm, case["transa"], case["transb"], ELEMS[case["elem"]][2])


def _batch_structures(case):
    top = np.random.default_rng(case["pattern"])
    out = []
    for p in range(case["count"]):
        n = int(top.integers(case["n_lo"], case["n_hi"] + 1))
        d = float(top.uniform(case["d_lo"], case["d_hi"]))
        rt, rm = _streams(case["pattern"] * 100003 + p + 1)
        r = G.tiling_uniform_int(n, case["b_lo"], case["b_hi"], rt)
        out.append(_Structure(r, r, r, *(G.mask_bernoulli(len(r), len(r), d, rm) for _ in range(2))))
    return out


# ---------------------------------------------------------------- values
def _uniform(count, dtype, gen):
    if dtype.is_complex:
        return torch.view_as_complex(torch.rand(count, 2, generator=gen, device="cuda", dtype=torch.float64) * 2 - 1)
    return torch.rand(count, generator=gen, device="cuda", dtype=dtype) * 2 - 1


def _decay(mask, rows, cols, align, count, gen, dtype):
    """Tile (i, j) holds N(0,1) exp(-|i-j|/2)."""
    i, j = np.nonzero(mask)
    size = rows.astype(np.int64)[i] * cols.astype(np.int64)[j]
    size = (size + align - 1) // align * align
    scale = torch.from_numpy(np.exp(-0.5 * np.abs(i - j))).cuda()
    scale = torch.repeat_interleave(scale, torch.from_numpy(size).cuda(), output_size=int(count))
    real = torch.float64 if dtype.is_complex else dtype
    shape = (count, 2) if dtype.is_complex else (count,)
    x = torch.randn(shape, generator=gen, device="cuda", dtype=real)
    x = torch.view_as_complex(x) if dtype.is_complex else x
    return x.mul_(scale.to(real))


def _arenas(case, st, gen):
    _, dtype, align = ELEMS[case["elem"]]
    if case["recipe"] == "banded_decay":
        ar, ac = (st.q, st.r) if st.transa else (st.r, st.q)
        br, bc = (st.c, st.q) if st.transb else (st.q, st.c)
        return (_decay(st.a_mask, ar, ac, align, st.a_len, gen, dtype),
                _decay(st.b_mask, br, bc, align, st.b_len, gen, dtype))
    return _uniform(st.a_len, dtype, gen), _uniform(st.b_len, dtype, gen)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _features(case, gen):
    """Rows as bsmm_plan_features gives them for split-mode units, and their log unit times."""
    n = case["rows"]
    u = torch.rand(n, 6, generator=gen, device="cuda", dtype=torch.float64)
    rows, cols = torch.floor(1 + 127 * u[:, 0] ** 0.2), torch.floor(1 + 31 * u[:, 1] ** 0.2)
    blocks = torch.floor(1 + 40 * u[:, 2])
    depth = torch.floor(blocks * (16 + 200 * u[:, 3]))
    steps, chunks = torch.floor(depth / 16 + 0.4 * blocks) + 1, torch.floor(depth / 32 + 0.5 * blocks) + 1
    flops = 2 * rows * cols * depth * (0.3 + 0.7 * u[:, 4])
    lg = lambda v: torch.log2(1 + v)  # noqa: E731
    tiles = torch.floor(1 + 3 * u[:, 5])
    X = torch.stack([lg(rows), lg(cols), lg(blocks), lg(depth), lg(steps), lg(flops), flops / (2 * 128 * 32 * 16 * steps),
                     torch.ones_like(rows), torch.ones_like(rows), lg(tiles), lg(torch.clamp(tiles - 1, min=1)),
                     lg(chunks)], dim=1)
    noise = torch.randn(n, generator=gen, device="cuda", dtype=torch.float64)
    t = torch.log(2000 + 450 * chunks + 700 * blocks + 300 * tiles) + 0.05 * noise
    return X.float().contiguous(), t.float().contiguous()


# ---------------------------------------------------------------- the four functions
def prepare(case, seed):
    gen = _gen(seed)
    if case["kind"] == "tile":
        m, n, k = case["m"], case["n"], case["k"]
        A, B, C = (_uniform(x, torch.float64, gen).reshape(s) for x, s in ((m * k, (m, k)), (k * n, (k, n)), (m * n, (m, n))))
        return {"case": case, "A": A, "B": B, "C": C}
    if case["kind"] == "fit":
        X, t = _features(case, gen)
        return {"case": case, "X": X, "t": t, "y": torch.empty_like(t), "seed": int(seed)}
    if case["kind"] == "batch":
        sts = _batch_structures(case)
        plans = [P.bsmm_plan(s.r, s.c, s.q, s.a_mask, s.b_mask, mode=MODES[case["mode"]], nslices=case["s"]) for s in sts]
        As, Bs = [_uniform(s.a_len, torch.float64, gen) for s in sts], [_uniform(s.b_len, torch.float64, gen) for s in sts]
        ends = np.cumsum([s.c_len for s in sts])
        C = torch.zeros(int(ends[-1]), dtype=torch.float64, device="cuda")
        Cs = [C[int(e) - s.c_len:int(e)] for e, s in zip(ends, sts)]
        ao, bo, co = ([_dev(x) for x in xs] for xs in ([s.a_off for s in sts], [s.b_off for s in sts], [s.c_off for s in sts]))
        batch = P.bsmm_batch_create(plans)
        n = len(plans)
        P.bsmm_batch_set_args(batch, [1.0] * n, As, ao, Bs, bo, [0.0] * n, Cs, co)
        return {"case": case, "batch": batch, "plans": plans, "C": C}
    st = _structure(case)
    elem, dtype, _ = ELEMS[case["elem"]]
    plan = P.bsmm_plan(st.r, st.c, st.q, st.a_mask, st.b_mask, mode=MODES[case["mode"]], nslices=case["s"],
                       cluster=case["cluster"], transa=case["transa"], transb=case["transb"],
                       split_scale=case["split_scale"], ksplit=case["ksplit"], elem=elem)
    A, B = _arenas(case, st, gen)
    C = _uniform(st.c_len, dtype, gen) if case["beta"] else torch.zeros(st.c_len, dtype=dtype, device="cuda")
    return {"case": case, "plan": plan, "A": A, "B": B, "C": C, "a_off": _dev(st.a_off), "b_off": _dev(st.b_off),
            "c_off": _dev(st.c_off)}


def run(state):
    case = state["case"]
    if case["kind"] == "tile":
        P.bsmm_split_tile_noalloc(case["m"], case["n"], case["k"], case["s"], case["alpha"], state["A"], state["B"],
                                  case["beta"], state["C"])
        return state["C"]
    if case["kind"] == "fit":
        # a fresh model, trained, and its predictions: what re-packing a plan by learned costs takes
        mlp = P.bsmm_mlp_create(state["seed"])
        loss = P.bsmm_mlp_fit(mlp, state["X"], state["t"], case["steps"], case["lr"])
        P.bsmm_mlp_predict(mlp, state["X"], state["y"])
        return {"loss": loss, "params": P.bsmm_mlp_get_params(mlp), "y": state["y"]}
    if case["kind"] == "batch":
        P.bsmm_batch_execute(state["batch"])
        return state["C"]
    execute = P.bsmm_execute_f32 if case["elem"] == "f32" else P.bsmm_execute
    execute(state["plan"], case["alpha"], state["A"], state["a_off"], state["B"], state["b_off"], case["beta"],
            state["C"], state["c_off"])
    return state["C"]


def _slice_products(case):
    return 1 if case["mode"] == "fp64" else case["s"] * (case["s"] + 1) // 2


def work(case):
    """Operands read once and C written once; the tensor-core (FP64) operations of the nonzero
    tile products: s(s+1)/2 slice products per multiplication in the split modes."""
    if case["kind"] == "tile":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 8.0 * (m * k + k * n + m * n * (2 if case["beta"] else 1)),
                "flops": 2.0 * m * n * k * case["s"] * (case["s"] + 1) / 2}
    if case["kind"] == "fit":
        per = 2.0 * (12 * 32 + 32 * 32 + 32)
        return {"bytes": 4.0 * case["rows"] * 14, "flops": case["rows"] * per * (3 * case["steps"] + 2)}
    if case["kind"] == "batch":
        sts = _batch_structures(case)
        return {"bytes": 8.0 * sum(sum(s.elements()) for s in sts),
                "flops": _slice_products(case) * sum(s.useful_flops() for s in sts)}
    st = _structure(case)
    a, b, c = st.elements()
    size = {"f64": 8.0, "f32": 4.0, "c128": 16.0}[case["elem"]]
    return {"bytes": size * (a + b + c * (2 if case["beta"] else 1)),
            "flops": st.useful_flops() * _slice_products(case) * (4 if case["elem"] == "c128" else 1)}


# ---------------------------------------------------------------- in 64 bits, by torch alone
def _wide(x):
    return x if x.is_complex() else x.double()


def _dense(arena, off, rows, cols, trans):
    """The stored matrix as a dense one, in its untransposed orientation (rows x cols tiling)."""
    u, v = (cols, rows) if trans else (rows, cols)  # the stored orientation
    uo, vo = (np.concatenate([[0], np.cumsum(x.astype(np.int64))]) for x in (u, v))
    out = torch.zeros(int(uo[-1]), int(vo[-1]), dtype=torch.complex128 if arena.is_complex() else torch.float64,
                      device="cuda")
    for i, j in zip(*np.nonzero(off >= 0)):
        o, m, n = int(off[i, j]), int(u[i]), int(v[j])
        out[int(uo[i]):int(uo[i + 1]), int(vo[j]):int(vo[j + 1])] = arena[o:o + m * n].view(m, n)
    return out.T if trans else out


def _exact_product(st, A, B, C0, alpha, beta):
    a = _dense(A, st.a_off, st.r, st.q, st.transa)
    b = _dense(B, st.b_off, st.q, st.c, st.transb)
    out = torch.zeros(C0.numel(), dtype=a.dtype, device="cuda")
    ro, co, qo = (np.concatenate([[0], np.cumsum(x.astype(np.int64))]) for x in (st.r, st.c, st.q))
    every = bool(st.am.all())
    for i in range(len(st.r)):
        js = np.nonzero(st.cs[i])[0]
        if not len(js):
            continue
        j0, j1 = int(co[js[0]]), int(co[js[-1] + 1])
        ai, bi = a[int(ro[i]):int(ro[i + 1])], b[:, j0:j1]
        if not every:  # the inner lines of the row's stored tiles
            inner = np.concatenate([np.arange(qo[k], qo[k + 1]) for k in np.nonzero(st.am[i])[0]])
            inner = torch.from_numpy(inner).cuda()
            ai, bi = ai[:, inner], bi[inner]
        ci = ai @ bi
        for j in js:
            o, m, n = int(st.c_off[i, j]), int(st.r[i]), int(st.c[j])
            t = alpha * ci[:, int(co[j]) - j0:int(co[j + 1]) - j0].reshape(-1)
            if beta:
                t = t + beta * _wide(C0[o:o + m * n])
            out[o:o + m * n] = t
    if beta:  # the alignment gaps between tiles are left as they were
        gap = torch.ones(C0.numel(), dtype=torch.bool, device="cuda")
        for i, j in zip(*np.nonzero(st.cs)):
            o = int(st.c_off[i, j])
            gap[o:o + int(st.r[i]) * int(st.c[j])] = False
        out = torch.where(gap, _wide(C0), out)
    return out


def _initial_params(seed):
    """The documented start of a model: splitmix64 from the seed, Box-Muller normals scaled by
    1/sqrt(fan-in) for the three weight arrays, zero biases; float32."""
    mask, state = (1 << 64) - 1, [seed & ((1 << 64) - 1)]

    def bits():
        state[0] = (state[0] + 0x9E3779B97F4A7C15) & mask
        z = state[0]
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        return (z ^ (z >> 31)) >> 11

    def normal():
        u1 = (bits() + 1.0) * 2.0 ** -53
        u2 = bits() * 2.0 ** -53
        return math.sqrt(-2.0 * math.log(u1)) * math.cos(6.283185307179586 * u2)

    w1 = [normal() / math.sqrt(12.0) for _ in range(384)]
    w2 = [normal() / math.sqrt(32.0) for _ in range(1024)]
    w3 = [normal() / math.sqrt(32.0) for _ in range(32)]
    return np.asarray(w1 + [0.0] * 32 + w2 + [0.0] * 32 + w3 + [0.0], np.float32)


def _exact_fit(case, seed):
    """Full-batch Adam on the mean squared standardised error of the 12-32-32-1 tanh network."""
    X32, t32 = _features(case, _gen(seed))
    w = torch.from_numpy(_initial_params(int(seed))).cuda().double()
    X, t = X32.double(), t32.double()
    mu, sd = X.mean(0), X.std(0, unbiased=False)
    mu, sd = mu.float().double(), torch.where(sd > 0, sd, torch.ones_like(sd)).float().double()
    ym, ys = t.mean().float().double(), t.std(unbiased=False).float().double()
    x, y = (X - mu) / sd, (t - ym) / ys
    n = len(y)
    cut = np.cumsum([0, 384, 32, 1024, 32, 32, 1])

    def layers(w):
        p = [w[cut[i]:cut[i + 1]] for i in range(6)]
        h1 = torch.tanh(x @ p[0].view(32, 12).T + p[1])
        h2 = torch.tanh(h1 @ p[2].view(32, 32).T + p[3])
        return p, h1, h2, h2 @ p[4] + p[5]

    m, v = torch.zeros_like(w), torch.zeros_like(w)
    for k in range(1, case["steps"] + 1):
        p, h1, h2, o = layers(w)
        dy = 2 * (o - y) / n
        d2 = dy[:, None] * p[4] * (1 - h2 * h2)
        d1 = (d2 @ p[2].view(32, 32)) * (1 - h1 * h1)
        g = torch.cat([(d1.T @ x).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0), h2.T @ dy, dy.sum()[None]])
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        w = w - case["lr"] * (m / (1 - 0.9 ** k)) / (torch.sqrt(v / (1 - 0.999 ** k)) + 1e-8)
    o = layers(w)[3]
    return {"loss": float(((o - y) ** 2).mean()), "params": w, "y": o * ys + ym}


def exact(case, seed):
    gen = _gen(seed)
    if case["kind"] == "tile":
        s = prepare(case, seed)
        return case["alpha"] * (s["A"] @ s["B"]) + case["beta"] * s["C"]
    if case["kind"] == "fit":
        return _exact_fit(case, seed)
    if case["kind"] == "batch":
        sts = _batch_structures(case)
        As, Bs = [_uniform(s.a_len, torch.float64, gen) for s in sts], [_uniform(s.b_len, torch.float64, gen) for s in sts]
        zero = [torch.zeros(s.c_len, dtype=torch.float64, device="cuda") for s in sts]
        return torch.cat([_exact_product(s, a, b, z, 1.0, 0.0) for s, a, b, z in zip(sts, As, Bs, zero)])
    st = _structure(case)
    _, dtype, _ = ELEMS[case["elem"]]
    A, B = _arenas(case, st, gen)
    C0 = _uniform(st.c_len, dtype, gen) if case["beta"] else torch.zeros(st.c_len, dtype=dtype, device="cuda")
    return _exact_product(st, A, B, C0, case["alpha"], case["beta"])

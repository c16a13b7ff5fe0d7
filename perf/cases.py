"""Work that users of this library have it do, as measurable cases.

Every case goes through the package's public calls on seeded synthetic tables: float32
rows of which 71 % of the columns are N(0, 1) and the rest integer codes 0..15, trees that
split on a uniform feature at a value met in the background, early leaves with probability
0.1, leaf values N(0, 0.1).  Kinds of cases:

  explain       phi of n consumer rows for a loaded ensemble whose background (or covers)
                is already set; rows in device memory, or in pinned host memory
  background    a new background of m rows, then phi of a few rows and the base value
  shards        pattern counts of a background shard, the background finished from the
                counts, then phi of a few rows
  batch         one graph launch over requests against several ensembles
  serve         a burst of host-memory requests to the continuous-batching server
  interactions  the F x F matrix of pairwise values of n rows
  global        FP64 column means of |phi| and phi of n explained rows

``exact`` restates the definitions in 64-bit torch: per leaf the table of cube values over
all (baseline pattern, consumer pattern) pairs, weighted with the exact baseline pattern
frequencies, looked up per consumer row and summed per feature.
"""
import math

import numpy as np
import torch

import paper_2511_09376_gb300 as wdf
from paper_2511_09376_gb300 import synth

DEV = "cuda:0"
GAUSS_SHARE = 0.71  # the KDD-Cup-99 mix after one-hot encoding: 90 of 127 columns
EARLY, LEAF_STD = 0.1, 0.1
BG_ROWS = 20_000   # background of the cases that measure the consumer side
FEW_ROWS = 64      # rows explained after a new background

# Most work a drawn case may ask for: rows x trees x leaves, and rows x features.
CAP_WORK = 1_000_000 * 200 * 64
CAP_CELLS = 130_000_000


def listed():
    return [
        # one prediction explained online on the paper's ensemble (100 trees of depth 6)
        dict(name="one_row", kind="explain", T=100, D=6, F=127, n=1),
        # a request of ordinary size on a mid-depth serving ensemble, Banzhaf values
        dict(name="request_777", kind="explain", T=500, D=7, F=112, n=777, metric="banzhaf"),
        # a test split explained at once: the paper's ensemble, 100,000 rows
        dict(name="mid", kind="explain", T=100, D=6, F=127, n=100_000),
        # a whole table explained: 200 trees, 1,000,000 rows of the KDD shape
        dict(name="large", kind="explain", T=200, D=6, F=127, n=1_000_000),
        # the deepest ensemble served (1000 trees of depth 8), split-precision background
        dict(name="deep", kind="explain", T=1000, D=8, F=134, n=20_011, precision="bf16x6"),
        # an export job: rows in pinned host memory, path-dependent values, shallow trees
        dict(name="host_path_dependent", kind="explain", T=150, D=5, F=127, n=150_001, where="host", freq="covers"),
        # a new background of the KDD shape (the other half of a Background SHAP run)
        dict(name="background_large", kind="background", T=200, D=6, F=127, m=1_000_000),
        # a background shard of a deep ensemble, counted and finished
        dict(name="shards_deep", kind="shards", T=300, D=8, F=134, m=60_013),
        # twelve models of different shapes explained in one launch
        dict(name="batch_ragged", kind="batch", count=12, T=400, rows=40_000, spec=4),
        # a burst of requests against three resident models
        dict(name="serve_burst", kind="serve", requests=24, T=400, rows=20_000, spec=5),
        # pairwise values: depth-6 ensemble, 127 x 127 per row
        dict(name="interactions", kind="interactions", T=200, D=6, F=127, n=4096),
        # global attribution of an explained table
        dict(name="global", kind="global", F=127, n=1_000_000),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _shape(rng, depths=(2, 8), trees=(10, 1000), feats=(20, 500)):
    D = rng.randint(*depths)
    return dict(T=_log(rng, *trees), D=D, F=rng.randint(*feats))


def draw(rng):
    kind = rng.choice(["explain", "explain", "explain", "background", "background", "shards", "batch", "serve",
                       "interactions", "global"])
    if kind == "explain":
        c = _shape(rng)
        top = min(1_000_000, CAP_WORK // (c["T"] << c["D"]), CAP_CELLS // c["F"])
        c.update(n=_log(rng, 1, max(1, top)), precision=rng.choice(["fp32", "fp32", "tf32x3", "bf16x6"]),
                 metric=rng.choice(["shapley", "shapley", "banzhaf"]), freq=rng.choice(["rows", "rows", "covers"]),
                 where=rng.choice(["device", "device", "host"]))
        if c["where"] == "host":
            c["n"] = min(c["n"], max(1, 20_000_000 // c["F"]))
    elif kind in ("background", "shards"):
        c = _shape(rng, trees=(10, 300))
        c["m"] = _log(rng, 1000, min(1_000_000, CAP_WORK // (c["T"] << c["D"]), CAP_CELLS // c["F"]))
        c["precision"] = rng.choice(["fp32", "fp32", "bf16x6"])
    elif kind == "batch":
        c = dict(count=rng.randint(2, 12), T=_log(rng, 20, 400), rows=_log(rng, 200, 40_000), spec=rng.randrange(1 << 20))
    elif kind == "serve":
        c = dict(requests=rng.randint(3, 32), T=_log(rng, 20, 400), rows=_log(rng, 20, 20_000),
                 spec=rng.randrange(1 << 20))
    elif kind == "interactions":
        c = _shape(rng, depths=(3, 8), trees=(10, 200), feats=(20, 200))
        c["n"] = _log(rng, 1, min(4096, 60_000_000 // (c["F"] * c["F"]), (4096 * 200 * 64) // (c["T"] << c["D"])))
    else:
        F = rng.randint(20, 500)
        c = dict(F=F, n=_log(rng, 1000, min(1_000_000, CAP_CELLS // F)))
    c["kind"] = kind
    return c


# ---- inputs ----

def _rows(seed, n, F):
    g = torch.Generator(device=DEV).manual_seed(seed)
    ng = int(round(GAUSS_SHARE * F))
    x = torch.empty((n, F), dtype=torch.float32, device=DEV)
    for r0 in range(0, n, 1 << 18):  # in pieces: the integer columns pass through int64
        r1 = min(n, r0 + (1 << 18))
        x[r0:r1, :ng] = torch.randn((r1 - r0, ng), generator=g, device=DEV)
        x[r0:r1, ng:] = torch.randint(0, 16, (r1 - r0, F - ng), generator=g, device=DEV).float()
    return x


class _Trees:
    """T trees in heap order, early leaves included.  feat/thr [T, 2^D - 1], value [T,
    2^(D+1) - 1]; state 0: no such node, 1: inner node, 2: leaf."""

    def __init__(self, seed, T, D, F, sample):
        rng = np.random.default_rng(seed)
        NI = (1 << D) - 1
        self.T, self.D, self.F = T, D, F
        self.feat = rng.integers(0, F, size=(T, NI))
        self.thr = sample[rng.integers(0, sample.shape[0], size=(T, NI)), self.feat].astype(np.float32)
        self.value = rng.normal(0.0, LEAF_STD, size=(T, 2 * NI + 1)).astype(np.float32)
        early = rng.random((T, NI)) < EARLY
        early[:, 0] = False
        self.state = np.zeros((T, 2 * NI + 1), np.int8)
        self.state[:, 0] = 1
        for d in range(1, D + 1):
            lo, hi = (1 << d) - 1, (1 << (d + 1)) - 1
            up = np.repeat(self.state[:, (lo - 1) // 2:(hi - 1) // 2] == 1, 2, axis=1)
            self.state[:, lo:hi] = np.where(up, 2 if d == D else np.where(early[:, lo:hi], 2, 1) if d < D else 2, 0)

    def ensemble(self):
        """The trees with their nodes numbered in heap order."""
        T, NI = self.T, self.feat.shape[1]
        there = self.state > 0
        num = np.cumsum(there, axis=1) - 1
        inner = self.state[:, :NI] == 1
        n_all = self.state.shape[1]
        feat, thr = np.full((T, n_all), -1, np.int32), np.zeros((T, n_all), np.float32)
        left, right = np.full((T, n_all), -1, np.int32), np.full((T, n_all), -1, np.int32)
        feat[:, :NI][inner] = self.feat[inner]
        thr[:, :NI][inner] = self.thr[inner]
        left[:, :NI][inner] = num[:, 1::2][inner]
        right[:, :NI][inner] = num[:, 2::2][inner]
        value = np.where(self.state == 2, self.value, np.float32(0))
        off = np.concatenate([[0], np.cumsum(there.sum(1))]).astype(np.int64)
        return synth.Ensemble(self.F, off, feat[there], thr[there], left[there], right[there], value[there])

    def covers(self, X):
        """Cover of every heap node: the rows of X that reach it, plus one per leaf."""
        T, D, NI = self.T, self.D, self.feat.shape[1]
        reach = torch.zeros((T, 2 * NI + 1), dtype=torch.float64, device=X.device)
        f, th = torch.from_numpy(self.feat).to(X.device), torch.from_numpy(self.thr).to(X.device)
        inner = torch.from_numpy(self.state[:, :NI] == 1).to(X.device)
        for t in range(T):
            left = (X[:, f[t]] < th[t]) & inner[t]
            here = torch.ones((X.shape[0], 1), dtype=torch.bool, device=X.device)
            for d in range(D + 1):
                reach[t, (1 << d) - 1:(1 << (d + 1)) - 1] = here.sum(0).double()
                if d < D:
                    lv, inn = left[:, (1 << d) - 1:(1 << (d + 1)) - 1], inner[t, (1 << d) - 1:(1 << (d + 1)) - 1]
                    here = torch.stack([here & lv, here & ~lv & inn], 2).reshape(X.shape[0], -1)
        cover = reach.cpu().numpy()
        cover = np.where(self.state == 2, cover + 1.0, 0.0)
        for v in range(NI - 1, -1, -1):
            cover[:, v] = np.where(self.state[:, v] == 1, cover[:, 2 * v + 1] + cover[:, 2 * v + 2], cover[:, v])
        return cover


def _model(seed, T, D, F, sample_rows=4096):
    return _Trees(seed, T, D, F, _rows(seed + 1, sample_rows, F).cpu().numpy())


def _load(ctx, trees, metric="shapley"):
    e = wdf.load_ensemble(ctx, trees.ensemble())
    if metric != "shapley":
        wdf.set_metric(e, metric)
    return e


def _several(case, count):
    """Shapes and row counts of the ensembles and requests of a batch or a burst."""
    rng = np.random.default_rng(case["spec"])
    shapes = [dict(T=max(5, int(round(case["T"] * math.exp(-2.5 * rng.random())))), D=2 + (i * 3 + int(rng.integers(0, 2))) % 7,
                   F=int(rng.integers(20, 301))) for i in range(count)]
    return shapes, rng


def _batch_plan(case):
    shapes, rng = _several(case, case["count"])
    reqs = [(i, max(1, int(round(case["rows"] * math.exp(-3.5 * rng.random()))))) for i in range(case["count"])]
    return shapes, reqs


def _serve_plan(case):
    shapes, rng = _several(case, 3)
    reqs = [(int(rng.integers(0, 3)), max(1, int(round(case["rows"] * math.exp(-7.0 * rng.random())))))
            for _ in range(case["requests"])]
    return shapes, reqs


def prepare(case, seed):
    kind, s = case["kind"], 1000 * seed
    if kind == "global":
        g = torch.Generator(device=DEV).manual_seed(s)
        # attributions of a sparse-ish model: per-column scales over two decades
        scale = torch.logspace(-3, -1, case["F"], device=DEV)
        phi = torch.randn((case["n"], case["F"]), generator=g, device=DEV) * scale + 0.1 * scale
        return dict(kind=kind, ctx=wdf.ctx_create(0), phi=phi)
    ctx = wdf.ctx_create(0)
    st = dict(kind=kind, ctx=ctx)
    if kind in ("batch", "serve"):
        shapes, reqs = _batch_plan(case) if kind == "batch" else _serve_plan(case)
        ens = []
        for i, sh in enumerate(shapes):
            e = _load(ctx, _model(s + 10 * i, **sh))
            wdf.set_background(e, _rows(s + 10 * i + 2, BG_ROWS, sh["F"]), "bf16x6")
            ens.append(e)
        rows = [_rows(s + 500 + j, n, shapes[i]["F"]) for j, (i, n) in enumerate(reqs)]
        if kind == "batch":
            st.update(batch=wdf.batch_create(ctx, ens), requests=[(i, C) for (i, _), C in zip(reqs, rows)])
        else:
            torch.cuda.synchronize()
            st["server"] = wdf.server_create(ctx, ens, device_budget_bytes=4 << 30, n_slots=4, max_wave=32)
            pinned = [(torch.empty(C.shape, pin_memory=True).copy_(C), torch.empty(C.shape, pin_memory=True)) for C in rows]
            st["requests"] = [(i, C.numpy(), phi.numpy()) for (i, _), (C, phi) in zip(reqs, pinned)]
            st["pinned"] = pinned
        return st
    T, D, F = case["T"], case["D"], case["F"]
    trees = _model(s, T, D, F)
    e = _load(ctx, trees, case.get("metric", "shapley"))
    st.update(e=e, precision=case.get("precision", "fp32"))
    if kind in ("background", "shards"):
        st.update(B=_rows(s + 2, case["m"], F), C=_rows(s + 3, FEW_ROWS, F))
        return st
    if case.get("freq", "rows") == "covers":
        cover = trees.covers(_rows(s + 2, 2000, F))
        wdf.set_covers(e, cover[trees.state > 0])
        wdf.set_path_dependent(e, st["precision"])
    else:
        wdf.set_background(e, _rows(s + 2, BG_ROWS, F), st["precision"])
    C = _rows(s + 3, case["n"], F)
    if case.get("where", "device") == "host":
        st["C"] = torch.empty(C.shape, pin_memory=True).copy_(C)
        st["out"] = torch.empty(C.shape, pin_memory=True)
    else:
        st["C"] = C
    return st


# ---- one pass ----

def run(st):
    kind = st["kind"]
    if kind == "explain":
        return wdf.explain(st["e"], st["C"], out=st.get("out"))
    if kind == "background":
        wdf.set_background(st["e"], st["B"], st["precision"])
        phi = wdf.explain(st["e"], st["C"])
        return {"phi": phi, "base": wdf.expected_value(st["e"])}
    if kind == "shards":
        counts = wdf.background_counts(st["e"], st["B"])
        wdf.set_background_counts(st["e"], counts, st["B"].shape[0], st["precision"])
        return {"counts": counts, "phi": wdf.explain(st["e"], st["C"])}
    if kind == "batch":
        return wdf.batch_explain(st["batch"], st["requests"])
    if kind == "serve":
        tickets = [wdf.server_submit(st["server"], i, C, phi=phi)[0] for i, C, phi in st["requests"]]
        for t in tickets:
            wdf.server_wait(st["server"], t)
        return [phi for _, _, phi in st["requests"]]
    if kind == "interactions":
        return wdf.explain_interactions(st["e"], st["C"])
    mean_abs, mean = wdf.global_attribution(st["ctx"], st["phi"])
    return {"mean_abs": mean_abs, "mean": mean}


# ---- work ----

def _nodes(T, D):
    """Expected inner nodes of T trees (a node of depth d is one with probability (1 - EARLY)^d)."""
    return T * sum((2 * (1 - EARLY)) ** d for d in range(D))


def _explain_work(T, D, F, n):
    # every row and phi once, every node (feature, threshold, children, value: 20 bytes) once;
    # a comparison and an addition per row and node
    nodes = _nodes(T, D)
    return 8.0 * n * F + 20.0 * 2 * nodes, 2.0 * n * nodes


def work(case):
    kind = case["kind"]
    if kind == "global":
        return {"bytes": 4.0 * case["n"] * case["F"] + 16.0 * case["F"], "flops": 3.0 * case["n"] * case["F"]}
    if kind in ("batch", "serve"):
        shapes, reqs = _batch_plan(case) if kind == "batch" else _serve_plan(case)
        got = [_explain_work(n=n, **shapes[i]) for i, n in reqs]
        return {"bytes": sum(b for b, _ in got), "flops": sum(f for _, f in got)}
    T, D, F = case["T"], case["D"], case["F"]
    if kind == "explain":
        b, f = _explain_work(T, D, F, case["n"])
        return {"bytes": b, "flops": f}
    if kind == "interactions":
        # the matrices written once; a comparison per node and an addition per (node, ancestor)
        pairs = T * sum(d * (2 * (1 - EARLY)) ** d for d in range(D))
        return {"bytes": 4.0 * case["n"] * F * (F + 1), "flops": case["n"] * (_nodes(T, D) + pairs)}
    b, f = _explain_work(T, D, F, FEW_ROWS)
    # a comparison per row and node and a count per row and leaf; the counts of a shard
    counts = 4.0 * T * (1 << (D - 2)) * (2 << D) if kind == "shards" else 0.0
    return {"bytes": b + 4.0 * case["m"] * F + counts, "flops": f + 2.0 * case["m"] * _nodes(T, D)}


# ---- the same values in 64 bits ----

class _Exact:
    """Complete trees for the 64-bit restatement: an early leaf moves down to depth D through
    nodes without a feature that send every row left."""

    def __init__(self, trees):
        T, D, NI = trees.T, trees.D, trees.feat.shape[1]
        self.T, self.D, self.F = T, D, trees.F
        state, value = trees.state.copy(), np.where(trees.state == 2, trees.value.astype(np.float64), 0.0)
        self.feat = np.where(state[:, :NI] == 1, trees.feat, -1)
        for v in range(NI):
            move = state[:, v] == 2
            state[:, 2 * v + 1][move] = 2
            value[:, 2 * v + 1] = np.where(move, value[:, v], value[:, 2 * v + 1])
        self.w = value[:, NI:]
        self.thr = trees.thr
        q, k = np.meshgrid(np.arange(1 << D), np.arange(D), indexing="ij")
        self.path = ((1 << D) + q >> (D - k)) - 1        # [leaf, depth] heap node
        self.turn = q >> (D - 1 - k) & 1                 # 1: the path goes right there

    def patterns(self, t, X):
        """[rows, leaves] pattern of every row at every leaf, root decision first."""
        D = self.D
        f = torch.from_numpy(np.maximum(self.feat[t], 0)).to(DEV)
        left = (X[:, f] < torch.from_numpy(self.thr[t]).to(DEV)) | torch.from_numpy(self.feat[t] < 0).to(DEV)
        p = torch.zeros((X.shape[0], 1), dtype=torch.int64, device=DEV)
        for d in range(D):
            l = left[:, (1 << d) - 1:(1 << (d + 1)) - 1].long()
            p = torch.stack([2 * p + l, 2 * p + 1 - l], 2).reshape(X.shape[0], -1)
        return p

    def counts(self, X, piece):
        """Rows per (tree, leaf, pattern), float64 [T, leaves, 2^D]."""
        K = 1 << self.D
        at = torch.arange(K, device=DEV) * K
        out = torch.zeros((self.T, K, K), dtype=torch.float64, device=DEV)
        for t in range(self.T):
            for r0 in range(0, X.shape[0], piece):
                idx = (self.patterns(t, X[r0:r0 + piece]) + at).reshape(-1)
                out[t] += torch.bincount(idx, minlength=K * K).reshape(K, K).double()
        return out

    def cover_freq(self, cover):
        """Path-dependent pattern frequencies of every leaf from the node covers."""
        T, D, NI = self.T, self.D, self.feat.shape[1]
        K = 1 << D
        r = np.ones((T, K, D))
        for k in range(D):
            h = self.path[:, k]
            child = 2 * h + 1 + self.turn[:, k]
            here = self.feat[:, h] >= 0
            r[:, :, k] = np.where(here, cover[:, child] / np.where(here, cover[:, h], 1.0), 1.0 - self.turn[:, k])
        r = torch.from_numpy(r).to(DEV)
        out = torch.ones((T, K, 1), dtype=torch.float64, device=DEV)
        for k in range(D):
            out = torch.stack([out * (1 - r[:, :, k:k + 1]), out * r[:, :, k:k + 1]], 3).reshape(T, K, -1)
        return out

    def _cube(self, first):
        """Literals of the cube of every (consumer pattern, baseline pattern): [D, K, K] masks
        of positive and negative variables (a variable sits at its first path position) and
        whether the cube can hold."""
        D, K = self.D, 1 << self.D
        p = torch.arange(K, device=DEV)
        bits = [(p >> (D - 1 - k)) & 1 for k in range(D)]
        pos = torch.zeros((D, K, K), dtype=torch.bool, device=DEV)
        neg = torch.zeros_like(pos)
        fine = torch.ones((K, K), dtype=torch.bool, device=DEV)
        for k in range(D):
            c, b = bits[k][:, None] == 1, bits[k][None, :] == 1
            fine &= c | b
            pos[first[k]] |= c & ~b
            neg[first[k]] |= ~c & b
        fine &= ~(pos & neg).any(0)
        return pos, neg, fine

    def value_table(self, first, metric):
        """[baseline pattern, consumer pattern, position] value of the cube's variables."""
        D = self.D
        pos, neg, fine = self._cube(first)
        a, b = pos.sum(0), neg.sum(0)
        fac = torch.tensor([float(math.factorial(i)) for i in range(D + 1)], dtype=torch.float64, device=DEV)
        if metric == "banzhaf":
            vp = 0.5 ** (a + b - 1).clamp(min=0).double()
            vn = -vp
        else:  # (a-1)! b! / (a+b)!, -a! (b-1)! / (a+b)!
            vp = fac[(a - 1).clamp(min=0)] * fac[b] / fac[a + b]
            vn = -fac[a] * fac[(b - 1).clamp(min=0)] / fac[a + b]
        v = torch.where(pos, vp, torch.where(neg, vn, torch.zeros_like(vp))) * fine
        return v.permute(2, 1, 0).contiguous()

    def pair_table(self, first):
        """[baseline pattern, consumer pattern, position pair] Shapley interaction values."""
        D = self.D
        pos, neg, fine = self._cube(first)
        a, b = pos.sum(0), neg.sum(0)
        fac = torch.tensor([float(math.factorial(i)) for i in range(D + 1)], dtype=torch.float64, device=DEV)
        f = lambda i: fac[i.clamp(min=0)]  # noqa: E731
        pp = f(a - 2) * f(b) / f(a + b - 1)
        nn = f(a) * f(b - 2) / f(a + b - 1)
        pn = -f(a - 1) * f(b - 1) / f(a + b - 1)
        out = []
        for i in range(D):
            for j in range(i + 1, D):
                v = torch.where(pos[i] & pos[j], pp, torch.where(neg[i] & neg[j], nn, torch.where(
                    (pos[i] & neg[j]) | (neg[i] & pos[j]), pn, torch.zeros_like(pp)))) * fine
                out.append(v)
        return torch.stack(out, 2).permute(1, 0, 2).contiguous()

    def signatures(self):
        """{first-occurrence positions: flat (tree, leaf) indices} of the leaves that count."""
        T, D = self.T, self.D
        pf = self.feat[:, self.path]                     # [T, leaves, D]
        pf = np.where(pf < 0, -1 - np.arange(D), pf)
        first = np.argmax(pf[..., :, None] == pf[..., None, :], axis=-1)
        code = (first * (8 ** np.arange(D))).sum(-1).reshape(-1)
        live = np.nonzero(self.w.reshape(-1) != 0.0)[0]
        order = live[np.argsort(code[live], kind="stable")]
        cuts = np.nonzero(np.diff(code[order]))[0] + 1
        flat = first.reshape(-1, D)
        return [(tuple(int(v) for v in flat[g[0]]), torch.from_numpy(g).to(DEV)) for g in np.split(order, cuts)]

    def lookup(self, freq, table, width):
        """[T, leaves, consumer pattern, width]: leaf weight x sum over baseline patterns."""
        K = 1 << self.D
        out = torch.zeros((self.T * K, K, width), dtype=torch.float64, device=DEV)
        flat, w = freq.reshape(-1, K), torch.from_numpy(self.w.reshape(-1)).to(DEV)
        for first, g in self.signatures():
            tab = table(first).reshape(K, K * width)
            for g0 in torch.split(g, 4096):
                out[g0] = ((flat[g0] * w[g0, None]) @ tab).reshape(-1, K, width)
        return out.reshape(self.T, K, K, width)

    def values(self, S, C, piece):
        K, D = 1 << self.D, self.D
        phi = torch.zeros((C.shape[0], self.F + 1), dtype=torch.float64, device=DEV)
        at = torch.arange(K, device=DEV) * K
        for t in range(self.T):
            col = torch.from_numpy(np.where(self.feat[t] < 0, self.F, self.feat[t])).to(DEV)
            St = S[t].reshape(K * K, D)
            for r0 in range(0, C.shape[0], piece):
                v = St[self.patterns(t, C[r0:r0 + piece]) + at]      # [rows, leaves, D]
                node = torch.cat([v[:, :, k].reshape(v.shape[0], 1 << k, -1).sum(2) for k in range(D)], 1)
                phi[r0:r0 + piece].index_add_(1, col, node)
        return phi[:, :self.F].contiguous()

    def pairs(self, S, C, piece):
        K, D, F = 1 << self.D, self.D, self.F
        out = torch.zeros((C.shape[0], F * F + 1), dtype=torch.float64, device=DEV)
        at = torch.arange(K, device=DEV) * K
        ij = [(i, j) for i in range(D) for j in range(i + 1, D)]
        for t in range(self.T):
            pf = self.feat[t][self.path]                 # [leaves, D]
            fi = np.stack([pf[:, i] for i, _ in ij], 1)
            fj = np.stack([pf[:, j] for _, j in ij], 1)
            keep = (fi >= 0) & (fj >= 0) & (fi != fj)
            up = torch.from_numpy(np.where(keep, fi * F + fj, F * F).reshape(-1)).to(DEV)
            dn = torch.from_numpy(np.where(keep, fj * F + fi, F * F).reshape(-1)).to(DEV)
            St = S[t].reshape(K * K, len(ij))
            for r0 in range(0, C.shape[0], piece):
                v = St[self.patterns(t, C[r0:r0 + piece]) + at]
                v = v.reshape(v.shape[0], -1)
                out[r0:r0 + piece].index_add_(1, up, v).index_add_(1, dn, v)
        return out[:, :F * F].reshape(-1, F, F).contiguous()


def _exact_values(trees, freq, C, metric="shapley"):
    x = _Exact(trees)
    S = x.lookup(freq(x), lambda first: x.value_table(first, metric), x.D)
    return x.values(S, C, max(1, (1 << 28) // (8 * x.D << x.D))), x


def _rows_freq(B):
    return lambda x: x.counts(B, max(1, (1 << 28) // (8 << x.D))) / B.shape[0]


def exact(case, seed):
    kind, s = case["kind"], 1000 * seed
    if kind == "global":
        phi = prepare(case, seed)["phi"].double()
        return {"mean_abs": phi.abs().mean(0), "mean": phi.mean(0)}
    if kind in ("batch", "serve"):
        shapes, reqs = _batch_plan(case) if kind == "batch" else _serve_plan(case)
        if sum((BG_ROWS + n) * shapes[i]["T"] << shapes[i]["D"] for i, n in reqs) > 6e9:
            return None
        out = []
        for j, (i, n) in enumerate(reqs):
            sh = shapes[i]
            B = _rows(s + 10 * i + 2, BG_ROWS, sh["F"])
            out.append(_exact_values(_model(s + 10 * i, **sh), _rows_freq(B), _rows(s + 500 + j, n, sh["F"]))[0])
        return out
    T, D, F = case["T"], case["D"], case["F"]
    trees = _model(s, T, D, F)
    metric = case.get("metric", "shapley")
    if kind == "interactions":
        if D > 6:
            return None
        x = _Exact(trees)
        S = x.lookup(_rows_freq(_rows(s + 2, BG_ROWS, F))(x), x.pair_table, D * (D - 1) // 2)
        return x.pairs(S, _rows(s + 3, case["n"], F), max(1, (1 << 28) // (8 * D * D << D)))
    if kind in ("background", "shards"):
        B, C = _rows(s + 2, case["m"], F), _rows(s + 3, FEW_ROWS, F)
        phi, x = _exact_values(trees, _rows_freq(B), C, metric)
        if kind == "shards":
            return {"counts": None, "phi": phi}
        base = 0.0  # mean output of the background rows
        for t in range(T):
            w = torch.from_numpy(x.w[t]).to(DEV)
            for r0 in range(0, B.shape[0], 1 << 17):
                hit = x.patterns(t, B[r0:r0 + (1 << 17)]) == (1 << D) - 1
                base += float((hit.sum(0).double() * w).sum()) / B.shape[0]
        return {"phi": phi, "base": base}
    C = _rows(s + 3, case["n"], F)
    if case.get("freq", "rows") == "covers":
        cover = trees.covers(_rows(s + 2, 2000, F))
        freq = lambda x: x.cover_freq(cover)  # noqa: E731
    else:
        freq = _rows_freq(_rows(s + 2, BG_ROWS, F))
    return _exact_values(trees, freq, C, metric)[0]

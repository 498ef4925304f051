"""Performance cases of the semiring SpGEMM library: what a user has it do, through its public
entry points (`paper_2106_14402_gb300.cb`), over the sizes it is used at.

Families (field "kind" of a case):
  spgemm    C = A.B of one product, exact sizing, validation on (the defaults of `cb.spgemm`)
  colbatch  a product formed in column batches under an output budget; the consumer keeps each batch
  batched   many independent products in one call; the consumer keeps each wave's output
  merge     the (+)-merge of k partial results
  spmspv    y^T = x^T A for a sparse frontier x
  predict   the learned sizer's inference: features of every row, then the predicted sizes
  grad      one training mini-batch of the learned sizer: loss and gradient
Matrices are generated on the device: R-MAT (0.57/0.19/0.19/0.05, symmetrised), Erdos-Renyi with a
fixed number of distinct columns per row, and block-clustered.  A case names its graph by a number
("graph"); the seed relabels its vertices and draws its values, so every seed gives other inputs of
the same size, with outputs of the same size.
"""
import math
import random

import torch

from paper_2106_14402_gb300 import cb, sizer

DEV = "cuda"
RMAT = (0.57, 0.19, 0.19)
VALUE_BYTES = {"plus_times_i64": (8, 8, 8), "plus_times_f64": (8, 8, 8), "min_plus_u32": (4, 4, 4),
               "or_and_bool": (1, 1, 1), "sel2nd_min_i32": (4, 4, 4), "maxw_label": (4, 4, 8)}


def listed():
    return [
        # the smallest call: one product whose rows are all small; latency, launches and the
        # synchronisations of a default call count (a frontier or a small block of a larger product)
        {"name": "er16k_i64", "kind": "spgemm", "family": "er", "n": 16384, "deg": 8,
         "semiring": "plus_times_i64"},
        # a small graph's square over (select2nd, min): a millisecond, all row tiers, host steps visible
        {"name": "rmat14_sel2nd", "kind": "spgemm", "family": "rmat", "scale": 14, "n": 1 << 14, "ef": 16,
         "semiring": "sel2nd_min_i32"},
        # the headline product in its three value types (A.A of an R-MAT graph, heavy rows)
        {"name": "rmat18_f64", "kind": "spgemm", "family": "rmat", "scale": 18, "n": 1 << 18, "ef": 16,
         "semiring": "plus_times_f64"},
        {"name": "rmat18_u32", "kind": "spgemm", "family": "rmat", "scale": 18, "n": 1 << 18, "ef": 16,
         "semiring": "min_plus_u32"},
        {"name": "rmat18_bool", "kind": "spgemm", "family": "rmat", "scale": 18, "n": 1 << 18, "ef": 16,
         "semiring": "or_and_bool"},
        # high compression ratio, rows of one size: a protein-similarity network squared (clustering)
        {"name": "blocks_f64", "kind": "spgemm", "family": "blocks", "n": 100003, "cluster": 256,
         "semiring": "plus_times_f64"},
        # output larger than its budget: learned batch count, each batch kept by the consumer
        {"name": "colbatch_sel2nd", "kind": "colbatch", "family": "rmat", "scale": 17, "n": 1 << 17, "ef": 32,
         "semiring": "sel2nd_min_i32", "sizing": "learned", "budget": 4 << 30},
        # many independent products of uneven sizes, half (min,+) u32, half (+,x) f64
        {"name": "batched_mixed", "kind": "batched", "count": 128, "plan": 7, "mode": "sync_free"},
        # the merge that follows the stages of a distributed product
        {"name": "merge8_f64", "kind": "merge", "k": 8, "scale": 16, "edges": 1 << 25,
         "semiring": "plus_times_f64"},
        # one step of a traversal (shortest paths) from a frontier of 16K vertices
        {"name": "spmspv_u32", "kind": "spmspv", "scale": 18, "n": 1 << 18, "ef": 16, "frontier": 16384,
         "semiring": "min_plus_u32", "bucket": False},
        # the sizing step that stands in for a symbolic pass
        {"name": "sizer_predict", "kind": "predict", "scale": 19, "n": 1 << 19, "ef": 16},
        # one mini-batch of the sizer's training
        {"name": "sizer_grad", "kind": "grad", "scale": 14, "rows": 8192},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    case = _draw(rng)
    return case if case["kind"] == "batched" else {**case, "graph": rng.randint(1, 10 ** 6)}


def _draw(rng):
    kind = rng.choice(["spgemm", "spgemm", "spgemm", "spgemm", "spgemm", "colbatch", "batched", "merge",
                       "spmspv", "predict", "grad"])
    graph = rng.choice(["min_plus_u32", "sel2nd_min_i32", "or_and_bool", "plus_times_i64"])
    if kind == "spgemm":
        sr = rng.choice(list(VALUE_BYTES))
        family = rng.choice(["er", "rmat", "rmat", "blocks"])
        more = {"semiring": sr}
        if sr == "or_and_bool":
            more["falses"] = rng.choice([0.0, 0.0, 0.1, 0.6])
        if family == "er":
            return {"kind": kind, "family": family, "n": _log_int(rng, 256, 150000), "deg": rng.randint(4, 64), **more}
        if family == "rmat":
            n = _log_int(rng, 1 << 10, 200000)
            return {"kind": kind, "family": family, "scale": (n - 1).bit_length(), "n": n,
                    "ef": rng.randint(4, 16), **more}
        return {"kind": kind, "family": family, "n": _log_int(rng, 2000, 100000),
                "cluster": rng.choice([64, 128, 200, 256]), **more}
    if kind == "colbatch":
        n = _log_int(rng, 1 << 14, 1 << 17)
        budget = int(8 * (n + 1) + rng.uniform(0.15, 0.4) * 12 * n * 6000)
        return {"kind": kind, "family": "rmat", "scale": (n - 1).bit_length(), "n": n, "ef": rng.randint(8, 24),
                "semiring": graph, "sizing": rng.choice(["exact", "learned"]), "budget": budget}
    if kind == "batched":
        return {"kind": kind, "count": _log_int(rng, 8, 120), "plan": rng.randint(100, 10 ** 6),
                "mode": rng.choice(["sync_free", "host"])}
    if kind == "merge":
        return {"kind": kind, "k": rng.randint(2, 12), "scale": rng.randint(12, 16),
                "edges": _log_int(rng, 1 << 16, 1 << 24), "semiring": rng.choice([graph, "plus_times_f64"])}
    if kind == "spmspv":
        n = _log_int(rng, 1 << 13, 1 << 18)
        return {"kind": kind, "scale": (n - 1).bit_length(), "n": n, "ef": rng.randint(4, 16),
                "frontier": _log_int(rng, 64, n // 2), "semiring": graph, "bucket": rng.random() < 0.3}
    if kind == "predict":
        n = _log_int(rng, 1 << 12, 1 << 19)
        return {"kind": kind, "scale": (n - 1).bit_length(), "n": n, "ef": rng.randint(4, 16)}
    return {"kind": "grad", "scale": 14, "rows": _log_int(rng, 500, 14000)}


# ---- matrices ------------------------------------------------------------------------------------

def _generator(seed, *tags):
    s = int(seed)
    for t in tags:
        s = (s * 1000003 + int(t) + 12345) % (1 << 62)
    return torch.Generator(device=DEV).manual_seed(s)


def _csr_of_keys(keys, nrows, ncols):
    keys = torch.unique(keys)
    rows = torch.div(keys, ncols, rounding_mode="floor")
    col = (keys - rows * ncols).to(torch.int32)
    rp = torch.zeros(nrows + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(torch.bincount(rows, minlength=nrows), 0)
    return rp, col


def _rmat_edges(g, scale, m):
    a, b, c = RMAT
    i = torch.zeros(m, dtype=torch.int64, device=DEV)
    j = torch.zeros(m, dtype=torch.int64, device=DEV)
    for _ in range(scale):
        u = torch.rand(m, generator=g, device=DEV)
        i = 2 * i + (u >= a + b)
        j = 2 * j + (((u >= a) & (u < a + b)) | (u >= a + b + c))
    return i, j


def _labels(seed, tag, n):
    return torch.randperm(n, generator=_generator(seed, 9, tag), device=DEV)


def _rmat(case):
    """Edges of the symmetrised R-MAT graph on n <= 2^scale vertices (the graph cut to n of them)."""
    scale, n = case["scale"], case["n"]
    g = _generator(case.get("graph", 0), 1, scale, n, case.get("ef", 16))
    i, j = _rmat_edges(g, scale, case.get("ef", 16) << scale)
    perm = torch.randperm(1 << scale, generator=g, device=DEV)
    i, j = perm[i], perm[j]
    keep = (i < n) & (j < n)
    i, j = i[keep], j[keep]
    return torch.cat([i, j]), torch.cat([j, i])


def _er(g, n, deg, row_label, col_label):
    """CSR with min(deg, n) distinct columns per row, rows and columns relabelled."""
    d = min(deg, n)
    u = torch.sort(torch.rand(n, d, generator=g, device=DEV, dtype=torch.float64), 1).values
    col = (u * (n - d + 1)).long().clamp_(max=n - d) + torch.arange(d, device=DEV)
    out = torch.empty_like(col)
    out[row_label] = torch.sort(col_label[col], 1).values
    return torch.arange(n + 1, device=DEV, dtype=torch.int64) * d, out.to(torch.int32).reshape(-1)


def _blocks(case):
    """Edges of clusters of consecutive vertices with half of their pairs linked and one random link per
    vertex, symmetrised."""
    n, cluster = case["n"], case["cluster"]
    g = _generator(case.get("graph", 0), 2, n, cluster)
    v = torch.arange(n, device=DEV)
    pick = torch.rand(n, cluster, generator=g, device=DEV) < 0.5
    i, k = pick.nonzero(as_tuple=True)
    j = torch.div(i, cluster, rounding_mode="floor") * cluster + k
    i, j = i[j < n], j[j < n]
    far = torch.randint(n, (n,), generator=g, device=DEV)
    return torch.cat([i, v, j, far]), torch.cat([j, far, i, v])


def _values(g, dtype, count, semiring, falses=0.0):
    if dtype == torch.float64:
        return torch.rand(count, generator=g, device=DEV, dtype=torch.float64)
    if dtype == torch.float32:
        return torch.rand(count, generator=g, device=DEV)
    if dtype == torch.uint8:  # graphs store true; with `falses`, some stored values are explicit false
        return (torch.rand(count, generator=g, device=DEV) >= falses).to(torch.uint8)
    hi = {"min_plus_u32": 256, "plus_times_i64": 11}.get(semiring, 1 << 30)
    v = torch.randint(1, hi, (count,), generator=g, device=DEV, dtype=torch.int64)
    return v.to(torch.int32).view(torch.uint32) if dtype == torch.uint32 else v.to(dtype)


def _pattern(case, seed, rows=True, cols=True):
    """CSR pattern of the case's graph, its rows and columns relabelled by the seed's labels."""
    n = case["n"]
    label, same = _labels(seed, 0, n), torch.arange(n, device=DEV)
    row, column = label if rows else same, label if cols else same
    if case.get("family", "rmat") == "er":
        return _er(_generator(case.get("graph", 0), 3, n, case["deg"]), n, case["deg"], row, column)
    i, j = _blocks(case) if case.get("family", "rmat") == "blocks" else _rmat(case)
    return _csr_of_keys(row[i] * n + column[j], n, n)


def _operands(case, seed):
    """(A, B) of C = A.A: one matrix, or its pattern with two value types.  In a column-batched product
    only A's rows are relabelled, so that every seed has the same output in each range of columns."""
    n, sr = case["n"], case["semiring"]
    ta, tb, _ = cb.OPERAND_DTYPES[sr]
    batched = case["kind"] == "colbatch"
    rp, col = _pattern(case, seed, cols=not batched)
    g = _generator(seed, 4)
    A = cb.DeviceCSR(n, n, rp, col, _values(g, ta, col.numel(), sr, case.get("falses", 0.0)))
    if batched:
        rp, col = _pattern(case, seed, rows=False, cols=False)
    if batched or sr in ("maxw_label", "sel2nd_min_i32"):
        return A, cb.DeviceCSR(n, n, rp, col, _values(g, tb, col.numel(), sr))
    return A, A


def _plan(case):
    """Shapes of the products of a batched call: n log-uniform in [256, 65536], degree in [4, 64]."""
    r = random.Random(case["plan"])
    out = []
    for i in range(case["count"]):
        out.append((_log_int(r, 256, 65536), r.randint(4, 64),
                    "min_plus_u32" if i < case["count"] // 2 else "plus_times_f64"))
    return out


def _batched_operand(case, seed, product, right, n, deg, sr):
    """A_i (rows relabelled by the product's first labels, columns by its second) or B_i (second, third)."""
    first, second = _labels(seed, 3 * product + right, n), _labels(seed, 3 * product + right + 1, n)
    rp, col = _er(_generator(case["plan"], 5, product, right), n, deg, first, second)
    g = _generator(seed, 5, product, right)
    if sr == "plus_times_f64":
        val = torch.rand(col.numel(), generator=g, device=DEV, dtype=torch.float64) * 2 - 1
    else:
        val = torch.randint(1, 1001, (col.numel(),), generator=g, device=DEV).to(torch.int32).view(torch.uint32)
    return cb.DeviceCSR(n, n, rp, col, val)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind in ("spgemm", "colbatch"):
        s["A"], s["B"] = _operands(case, seed)
        if kind == "colbatch" and case["sizing"] == "learned":
            s["mlp"] = sizer.load()[0]
    elif kind == "batched":
        plan = _plan(case)
        s["srs"] = [sr for _, _, sr in plan]
        s["As"] = [_batched_operand(case, seed, i, 0, n, d, sr) for i, (n, d, sr) in enumerate(plan)]
        s["Bs"] = [_batched_operand(case, seed, i, 1, n, d, sr) for i, (n, d, sr) in enumerate(plan)]
    elif kind == "merge":
        n = 1 << case["scale"]
        rows, cols = _labels(seed, 0, n), _labels(seed, 1, n)
        s["parts"] = []
        for p in range(case["k"]):
            i, j = _rmat_edges(_generator(case.get("graph", 0), 6, p), case["scale"], case["edges"])
            rp, col = _csr_of_keys(rows[i] * n + cols[j], n, n)
            g = _generator(seed, 6, p)
            dt = cb.OPERAND_DTYPES[case["semiring"]][2]
            s["parts"].append(cb.DeviceCSR(n, n, rp, col, _values(g, dt, col.numel(), case["semiring"])))
    elif kind == "spmspv":
        s["A"], _ = _operands(case, seed)
        g = _generator(seed, 7)
        front = torch.randperm(case["n"], generator=_generator(case.get("graph", 0), 7), device=DEV)
        s["idx"] = _labels(seed, 0, case["n"])[front[:case["frontier"]]].to(torch.int32)
        s["val"] = _values(g, cb.OPERAND_DTYPES[case["semiring"]][0], case["frontier"], case["semiring"])
    elif kind == "predict":
        rp, col = _pattern(case, seed)
        s["A"] = cb.DeviceCSR(case["n"], case["n"], rp, col, torch.ones(col.numel(), dtype=torch.uint8, device=DEV))
        s["mlp"] = sizer.load()[0]
    else:  # grad: rows of a training product with their exact sizes
        n = 1 << case["scale"]
        rp, col = _pattern({**case, "n": n}, seed)
        A = cb.DeviceCSR(n, n, rp, col, torch.ones(col.numel(), dtype=torch.uint8, device=DEV))
        feat, nnz = cb.row_features(A, A), cb.row_nnz(A, A)
        pick = torch.randint(n, (case["rows"],), generator=_generator(seed, 8), device=DEV)
        s["feat"], s["nnz"] = feat[pick].contiguous(), nnz[pick].contiguous()
        s["mlp"] = sizer.load()[0]
    return s


def _plain(v):
    return v.view(torch.int32) if v.dtype == torch.uint32 else v


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "spgemm":
        C = cb.spgemm(case["semiring"], s["A"], s["B"])
        return C.row_ptr, C.col, _plain(C.val)
    if kind == "colbatch":
        bounds, rps, cols, vals = [], [], [], []

        def keep(batch, lo, hi, Cb):
            bounds.append((lo, hi))
            rps.append(Cb.row_ptr.clone())
            cols.append(Cb.col.clone())
            vals.append(_plain(Cb.val).clone())

        cb.spgemm_column_batches(case["semiring"], s["A"], s["B"], case["budget"], keep, sizing=case["sizing"],
                                 mlp=s.get("mlp"))
        return torch.tensor(bounds), rps, cols, vals
    if kind == "batched":
        waves = []

        def keep(wave, first, end, Cw):
            waves.append((first, end, Cw.row_ptr.clone(), Cw.col.clone(), _plain(Cw.val).clone()))

        cb.spgemm_batched(s["srs"], s["As"], s["Bs"], keep, mode=case["mode"])
        return waves
    if kind == "merge":
        C = cb.merge(case["semiring"], s["parts"])
        return C.row_ptr, C.col, _plain(C.val)
    if kind == "spmspv":
        idx, val = cb.spmspv(case["semiring"], s["A"], s["idx"], s["val"], bucket=case["bucket"])
        return idx, _plain(val)
    if kind == "predict":
        feat = cb.row_features(s["A"], s["A"])
        z, pred = s["mlp"].predict(feat, s["A"].ncols)
        return feat, z, pred
    return s["mlp"].grad(s["feat"], s["nnz"], 0.9)


# ---- work: each input read once, each output written once ----------------------------------------

def _csr_bytes(rows, nnz, value):
    return 8 * (rows + 1) + nnz * (4 + value)


def work(case):
    kind = case["kind"]
    if kind in ("spgemm", "colbatch"):
        rp, col = _pattern(case, 1)
        n = case["n"]
        A = cb.DeviceCSR(n, n, rp, col, torch.ones(col.numel(), dtype=torch.uint8, device=DEV))
        flops = int(cb.row_stats(A, A)[0].sum())
        out = int(cb.row_nnz(A, A).sum())
        va, vb, vc = VALUE_BYTES[case["semiring"]]
        two = vb * col.numel() if case["semiring"] in ("maxw_label", "sel2nd_min_i32") else 0
        a_val = 0 if case["semiring"] == "sel2nd_min_i32" else va
        return {"bytes": _csr_bytes(n, col.numel(), a_val) + two + _csr_bytes(n, out, vc), "flops": 2 * flops}
    if kind == "batched":
        nbytes = flops = 0
        for n, d, sr in _plan(case):
            v = VALUE_BYTES[sr][0]
            prods = n * d * d
            out = n * n * (1 - (1 - d / n) ** d)  # expected distinct columns
            nbytes += 2 * _csr_bytes(n, n * d, v) + _csr_bytes(n, int(out), v)
            flops += 2 * prods
        return {"bytes": nbytes, "flops": flops}
    if kind == "merge":
        parts = prepare(case, 1)["parts"]
        v = VALUE_BYTES[case["semiring"]][2]
        n = parts[0].nrows
        rows = [torch.repeat_interleave(torch.arange(n, device=DEV), p.row_ptr[1:] - p.row_ptr[:-1]) * n + p.col.long()
                for p in parts]
        out = torch.unique(torch.cat(rows)).numel()
        return {"bytes": sum(_csr_bytes(n, p.nnz, v) for p in parts) + _csr_bytes(n, out, v),
                "flops": sum(p.nnz for p in parts)}
    if kind == "spmspv":
        s = prepare(case, 1)
        lens = (s["A"].row_ptr[1:] - s["A"].row_ptr[:-1])[s["idx"].long()]
        prods = int(lens.sum())
        v = VALUE_BYTES[case["semiring"]][0]
        out = cb.spmspv(case["semiring"], s["A"], s["idx"], s["val"])[0].numel()
        return {"bytes": case["frontier"] * (4 + v + 16) + (prods + out) * (4 + v), "flops": 2 * prods}
    if kind == "predict":
        rp, col = _pattern(case, 1)
        return {"bytes": _csr_bytes(case["n"], col.numel(), 0) + case["n"] * (16 + 4 + 8),
                "flops": case["n"] * 2 * (3 * 64 + 64 * 64 + 64)}
    return {"bytes": case["rows"] * (16 + 8) + 2 * 4 * 4481, "flops": case["rows"] * 6 * (3 * 64 + 64 * 64 + 64)}


# ---- 64-bit results without the library ----------------------------------------------------------

def _product_f64(A, B):
    """Values of A.B in CSR order (columns ascending), each the plain sum of its products in 64 bits."""
    n, k = A.nrows, B.ncols
    lens = B.row_ptr[1:] - B.row_ptr[:-1]
    a_rows = torch.repeat_interleave(torch.arange(n, device=DEV), A.row_ptr[1:] - A.row_ptr[:-1])
    per = lens[A.col.long()]
    ends = torch.cumsum(per, 0)
    rows_at = max(1, (1 << 29) // k)
    vals = []
    for r0 in range(0, n, rows_at):
        r1 = min(n, r0 + rows_at)
        acc = torch.zeros((r1 - r0) * k, dtype=torch.float64, device=DEV)
        hit = torch.zeros((r1 - r0) * k, dtype=torch.bool, device=DEV)
        p, p_end = int(A.row_ptr[r0]), int(A.row_ptr[r1])
        while p < p_end:
            done = int(ends[p - 1]) if p else 0
            q = int(torch.searchsorted(ends, torch.tensor(done + (1 << 27), device=DEV)))
            q = min(p_end, max(q, p + 1))
            own = torch.repeat_interleave(torch.arange(p, q, device=DEV), per[p:q])
            first = ends[own] - per[own]
            at = B.row_ptr[A.col[own].long()] + torch.arange(own.numel(), device=DEV) + done - first
            key = (a_rows[own] - r0) * k + B.col[at].long()
            acc.index_add_(0, key, A.val[own] * B.val[at])
            hit[key] = True
            p = q
        vals.append(acc[hit])
        del acc, hit
    return torch.cat(vals)


def _sizer_forward(mlp, feat):
    """The predictor as documented (bf16 inputs, weights and activations), sums in 64 bits."""
    def bf(t):
        return t.to(torch.bfloat16).double()

    params, norm, _ = mlp.get()
    p = torch.from_numpy(params).to(DEV)
    norm = torch.from_numpy(norm).to(DEV).double()
    W1, b1, W2, b2, w3, b3 = torch.split(p, [192, 64, 4096, 64, 64, 1])
    f = feat.double()
    lw = torch.log2(f[:, 3].clamp(min=1.0))
    ln = torch.stack([torch.log2(1 + f[:, 0]), torch.log2(1 + f[:, 1]) - lw, torch.log2(1 + f[:, 2]) - lw], 1)
    x = bf((ln - norm[:3]) / norm[3:])
    W1, W2, w3 = bf(W1.view(64, 3)), bf(W2.view(64, 64)), bf(w3)
    h1 = bf((x @ W1.T + b1.double()).clamp(min=0))
    h2 = bf((h1 @ W2.T + b2.double()).clamp(min=0))
    return x, W2, w3, h1, h2, h2 @ w3 + b3.double()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("spgemm", "merge") and case["semiring"] != "plus_times_f64":
        return None  # whole numbers
    if kind == "spgemm":
        A, B = _operands(case, seed)
        return None, None, _product_f64(A, B)
    if kind == "merge":
        parts = prepare(case, seed)["parts"]
        n = parts[0].nrows
        keys = torch.cat([torch.repeat_interleave(torch.arange(n, device=DEV), p.row_ptr[1:] - p.row_ptr[:-1]) * n
                          + p.col.long() for p in parts])
        keys, at = torch.unique(keys, return_inverse=True)
        out = torch.zeros(keys.numel(), dtype=torch.float64, device=DEV)
        return None, None, out.index_add_(0, at, torch.cat([p.val for p in parts]))
    if kind == "batched":
        s = prepare(case, seed)
        vals = [_product_f64(a, b) for a, b, sr in zip(s["As"], s["Bs"], s["srs"]) if sr == "plus_times_f64"]
        waves = [(None,) * 5] if case["count"] // 2 else []
        return waves + [(None, None, None, None, torch.cat(vals))]
    if kind == "predict":
        s = prepare(case, seed)
        rp, col, n = s["A"].row_ptr, s["A"].col, s["A"].nrows
        lens = rp[1:] - rp[:-1]
        rows = torch.repeat_interleave(torch.arange(n, device=DEV), lens)
        of = lens[col.long()]
        flops = torch.zeros(n, dtype=torch.int64, device=DEV).index_add_(0, rows, of)
        maxb = torch.zeros(n, dtype=torch.int64, device=DEV).scatter_reduce_(0, rows, of, "amax")
        feat = torch.stack([lens, flops, maxb, torch.full_like(lens, n)], 1).double()
        return feat, _sizer_forward(s["mlp"], feat.float())[-1], None
    if kind == "grad":
        s = prepare(case, seed)
        x, W2, w3, h1, h2, z = _sizer_forward(s["mlp"], s["feat"])
        fl = s["feat"][:, 1].double()
        live = fl > 0
        cnt = max(int(live.sum()), 1)
        ratio = torch.where(live, s["nnz"].double() / fl.clamp(min=1), torch.ones_like(fl))
        e = torch.log2(ratio) - torch.nn.functional.logsigmoid(z) / math.log(2)
        loss = torch.where(live, torch.where(e >= 0, 0.9 * e, -0.1 * e), torch.zeros_like(e)).sum() / cnt
        slope = torch.where(e >= 0, torch.full_like(e, 0.9), torch.full_like(e, -0.1))
        dz = torch.where(live, -slope * torch.sigmoid(-z) / math.log(2), torch.zeros_like(e)) / cnt
        d2 = dz[:, None] * w3 * (h2 > 0)
        d1 = (d2 @ W2) * (h1 > 0)
        g = [(d1.T @ x).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0), h2.T @ dz, dz.sum()[None]]
        return torch.cat(g), loss[None]
    return None

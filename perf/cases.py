"""Performance cases: calls that programs using this package make, through its public entry points.

Every case is one call (or, for the conversions, one pair of calls) on a handle, over the range the
package serves: one lattice from a single site to 64^4 sites, every storage type, representation
and memory layout, plain and FP32-pair arithmetic, the adjacent products, the batch of uneven
lattices, the conversions in and out of the benchmark's format, and buffers in host memory.

``tuned`` cases install the package's measured launch shapes on the handle first, as bench.py does;
the others use a handle as it comes, as in the package's usage example.
"""
import ctypes

import numpy as np
import torch

import paper_2103_00571_gb300 as su3
from paper_2103_00571_gb300 import tune

DTYPES = {"f64": su3.F64, "f32": su3.F32, "f16": su3.F16, "bf16": su3.BF16}
TORCH = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
REAL = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}
LAYOUTS = {"aos": su3.AOS, "aosoa32": su3.AOSOA32, "soa": su3.SOA}
ARITHS = {"native": su3.NATIVE, "f32pair": su3.F32PAIR}
REPRS = {"full": su3.FULL18, "2row": su3.TWOROW12}
ELEMS = {"full": 9, "2row": 6}
OPS = {"nn": su3.OP_NN, "na": su3.OP_NA, "an": su3.OP_AN}
MAX_SITES = 64 ** 4


def _mult(name, sites, dtype="f64", a="full", c="full", layout="aos", arith="native", stride=0, op="nn", tuned=True):
    return {"name": name, "kind": "mult", "sites": sites, "dtype": dtype, "a": a, "c": c, "layout": layout,
            "arith": arith, "stride": stride, "op": op, "tuned": tuned}


def listed():
    return [
        # a small lattice, called in a loop (the correctness configuration): latency
        _mult("f64_L8", 8 ** 4, tuned=False),
        # the benchmark's own size, straight from the usage example
        _mult("f64_L32", 32 ** 4, tuned=False),
        # the headline workload: larger than any cache
        _mult("f64_L64", 64 ** 4),
        # the benchmark's padded 640-byte Site structure, as its C code lays it out
        _mult("f64_site640_L32", 32 ** 4, stride=640),
        # FP64 storage at the FP32 units' speed
        _mult("f64_pair_L48", 48 ** 4, arith="f32pair"),
        # compressed gauge links expanded on the fly (a third fewer bytes read), at an odd extent
        _mult("f64_2row_to_full_21", 21 ** 4, a="2row"),
        # single precision in the vector-friendly layout, a ragged number of links, handle as it comes
        _mult("f32_aosoa32_ragged", 1000003, dtype="f32", layout="aosoa32", tuned=False),
        # reduced storage at full size (50 iterations of this are the precision study)
        _mult("bf16_L64", 64 ** 4, dtype="bf16"),
        # the links applied to colour vectors (the other core product of lattice codes)
        {"name": "f64_matvec_L32", "kind": "matvec", "sites": 32 ** 4, "dtype": "f64", "arith": "native",
         "adjoint": False, "tuned": True},
        # 96 small lattices of mixed precision in one launch, replayed
        {"name": "batch96", "kind": "batch", "lattices": 96, "max_extent": 24, "mix": 2103, "arith": "native", "tuned": True},
        # into a reduced form and back, the set-up of every reduced-precision run
        {"name": "convert_f16_soa_L40", "kind": "convert", "sites": 40 ** 4, "dtype": "f16", "a": "full",
         "layout": "soa", "tuned": False},
        # data that lives in pinned host memory
        {"name": "host_f64_L24", "kind": "host", "sites": 24 ** 4, "dtype": "f64", "arith": "native", "tuned": False},
    ]


def _log_sites(rng, hi):
    return max(1, int(round(2.0 ** rng.uniform(0.0, np.log2(hi)))))


def draw(rng):
    tuned = rng.random() < 0.5
    kind = rng.choice(["mult"] * 6 + ["matvec", "batch", "convert", "host"])
    dtype = rng.choice(["f64", "f64", "f64", "f32", "f16", "bf16"])
    arith = rng.choice(["native", "native", "f32pair"]) if dtype == "f64" else "native"
    sites = _log_sites(rng, MAX_SITES)
    if kind == "mult":
        a, c = rng.choice([("full", "full"), ("full", "full"), ("2row", "2row"), ("2row", "full")])
        layout = rng.choice(["aos", "aos", "aosoa32", "soa"])
        op, stride = "nn", 0
        if layout == "aos":
            if a == "full":
                op = rng.choice(["nn", "nn", "na", "an"])
            if dtype == "f64" and a == c and rng.random() < 0.3:
                stride = 640
                sites = min(sites, MAX_SITES // 2)
        case = _mult("", sites, dtype, a, c, layout, arith, stride, op, tuned)
        del case["name"]
        return case
    if kind == "matvec":
        return {"kind": kind, "sites": sites, "dtype": dtype, "arith": arith, "adjoint": rng.random() < 0.5,
                "tuned": tuned}
    if kind == "batch":
        return {"kind": kind, "lattices": rng.randint(1, 96), "max_extent": 2 * rng.randint(2, 12),
                "mix": rng.randrange(1 << 20), "arith": rng.choice(["native", "f32pair"]), "tuned": tuned}
    if kind == "convert":
        return {"kind": kind, "sites": min(sites, MAX_SITES // 4), "dtype": dtype, "a": rng.choice(["full", "full", "2row"]),
                "layout": rng.choice(["aos", "aosoa32", "soa"]), "tuned": False}
    return {"kind": kind, "sites": min(sites, MAX_SITES // 16), "dtype": dtype, "arith": arith, "tuned": tuned}


# ---- inputs: random SU(3) matrices (Gram-Schmidt on two normal rows, third row their cross product) ----

CHUNK = 1 << 20  # links


def _su3(gen, n):
    """n random SU(3) matrices as float64 [n, 3, 3, 2]."""
    out = torch.empty(n, 3, 3, 2, dtype=torch.float64, device="cuda")
    for i in range(0, n, CHUNK):
        m = min(CHUNK, n - i)
        z = torch.view_as_complex(torch.randn(m, 2, 3, 2, dtype=torch.float64, device="cuda", generator=gen))
        u = z[:, 0] / torch.linalg.vector_norm(z[:, 0], dim=1, keepdim=True)
        v = z[:, 1] - (u.conj() * z[:, 1]).sum(1, keepdim=True) * u
        v = v / torch.linalg.vector_norm(v, dim=1, keepdim=True)
        w = torch.linalg.cross(u, v).conj()
        out[i:i + m] = torch.view_as_real(torch.stack([u, v, w], 1))
    return out


def _gen(seed, part=0):
    return torch.Generator(device="cuda").manual_seed(1000003 * (seed + 1) + part)


def _links(seed, sites, part=0):
    """(a [4 * sites, 3, 3, 2] on the GPU, b: 72 doubles on the host) of one lattice."""
    g = _gen(seed, part)
    b = _su3(g, 4).cpu().numpy().reshape(72)
    return _su3(g, 4 * sites), b


def _to_layout(x, layout, dtype, sites, stride):
    """Links [n, elements, 2] as the array the package takes (elements 9 full, 6 two-row)."""
    n, ne = x.shape[0], x.shape[1]
    x = x.to(dtype)
    if layout == "soa":
        return x.permute(1, 0, 2).contiguous().view(-1)
    if layout == "aosoa32":
        blocks = (n + 31) // 32
        y = torch.zeros(blocks * 32, ne, 2, dtype=dtype, device=x.device)
        y[:n] = x
        return y.view(blocks, 32, ne, 2).permute(0, 2, 1, 3).contiguous().view(-1)
    if stride:
        y = torch.zeros(sites, stride // x.element_size(), dtype=dtype, device=x.device)
        y[:, :4 * ne * 2] = x.reshape(sites, -1)
        return y.view(-1)
    return x.reshape(-1)


def _handle(case):
    h = su3.Handle(0)
    if case["tuned"]:
        tune.apply_cached(h)
    return h


def _descs(case):
    args = LAYOUTS[case["layout"]], case["sites"], case["stride"], ARITHS[case["arith"]]
    dt = DTYPES[case["dtype"]]
    return su3.Desc(dt, REPRS[case["a"]], *args), su3.Desc(dt, REPRS[case["c"]], *args)


def _batch_lattices(case):
    """Sites and storage types of a batch: like the benchmark's, extents even, from 4 up."""
    rng = np.random.default_rng(case["mix"])
    ext = 4 + 2 * rng.integers(0, case["max_extent"] // 2 - 1, size=(case["lattices"], 4))
    return [(int(np.prod(e)), "f64" if k % 2 == 0 else "f32") for k, e in enumerate(ext)]


def prepare(case, seed):
    kind = case["kind"]
    h = _handle(case)
    st = {"kind": kind, "h": h}
    if kind == "batch":
        lattices = _batch_lattices(case)
        items, keep = [], []
        # the results of all lattices of a storage type lie in one pool
        outs = {t: torch.zeros(sum(72 * n for n, d in lattices if d == t), dtype=TORCH[t], device="cuda")
                for t in ("f64", "f32") if any(d == t for _, d in lattices)}
        at = dict.fromkeys(outs, 0)
        for k, (sites, dtype) in enumerate(lattices):
            a, b = _links(seed, sites, k)
            a = a.to(TORCH[dtype]).reshape(-1)
            c = outs[dtype][at[dtype]:at[dtype] + 72 * sites]
            at[dtype] += 72 * sites
            d = su3.Desc(DTYPES[dtype], su3.FULL18, su3.AOS, sites, 0,
                         ARITHS[case["arith"]] if dtype == "f64" else su3.NATIVE)
            items.append(su3.BatchItem(d, a.data_ptr(), c.data_ptr(), (ctypes.c_double * 72)(*b)))
            keep.append(a)
        st.update(items=items, keep=keep, outs=list(outs.values()))
        return st
    sites, dtype = case["sites"], TORCH[case["dtype"]]
    a, b = _links(seed, sites)
    if kind == "mult":
        da, dc = _descs(case)
        a = a.view(4 * sites, 9, 2)[:, :ELEMS[case["a"]]]
        st["a"] = _to_layout(a, case["layout"], dtype, sites, case["stride"])
        st["c"] = torch.zeros(su3.array_bytes(dc) // REAL[case["dtype"]], dtype=dtype, device="cuda")
        st.update(b=b, da=da, dc=dc, op=OPS[case["op"]])
    elif kind == "matvec":
        st["a"] = a.to(dtype).reshape(-1)
        st["v"] = b.reshape(4, 3, 3, 2)[:, 0].copy()
        st["w"] = torch.zeros(sites * 24, dtype=dtype, device="cuda")
        st["da"] = su3.Desc(DTYPES[case["dtype"]], su3.FULL18, su3.AOS, sites, 0, ARITHS[case["arith"]])
        st["adjoint"] = case["adjoint"]
    elif kind == "convert":
        st["a"] = a.reshape(-1)
        st["d"] = su3.Desc(DTYPES[case["dtype"]], REPRS[case["a"]], LAYOUTS[case["layout"]], sites)
        st["form"] = torch.zeros(su3.array_bytes(st["d"]) // REAL[case["dtype"]], dtype=dtype, device="cuda")
        st["back"] = torch.zeros(sites * 72, dtype=torch.float64, device="cuda")
    else:
        st["a"] = a.to(dtype).reshape(-1).cpu().pin_memory()
        st["c"] = torch.zeros(sites * 72, dtype=dtype).pin_memory()
        st["b"] = b
        st["d"] = su3.Desc(DTYPES[case["dtype"]], su3.FULL18, su3.AOS, sites, 0, ARITHS[case["arith"]])
    return st


def run(st):
    h, kind = st["h"], st["kind"]
    if kind == "mult":
        if st["op"] == su3.OP_NN:
            h.mult(st["da"], st["a"], st["b"], st["dc"], st["c"])
        else:
            h.mult_op(st["op"], st["da"], st["a"], st["b"], st["dc"], st["c"])
        return st["c"]
    if kind == "matvec":
        h.mat_vec(st["da"], st["a"], st["v"], st["w"], adjoint=st["adjoint"])
        return st["w"]
    if kind == "batch":
        h.mult_batched(st["items"], use_graph=True)
        return st["outs"]
    if kind == "convert":
        h.pack(st["a"], st["d"], st["form"])
        h.unpack(st["d"], st["form"], st["back"])
        return [st["form"], st["back"]]
    h.mult_host(st["d"], st["a"], st["b"], st["d"], st["c"])
    return st["c"]


def work(case):
    kind = case["kind"]
    if kind == "batch":
        lattices = _batch_lattices(case)
        return {"bytes": sum(n * 144 * REAL[d] for n, d in lattices), "flops": sum(n * 864 for n, _ in lattices)}
    sites, real = case["sites"], REAL[case["dtype"]]
    if kind == "mult":
        rows_out = {"full": 864, "2row": 576}[case["c"]]
        rebuild = 4 * 3 * 14 if case["a"] != case["c"] else 0
        return {"bytes": sites * 8 * real * (ELEMS[case["a"]] + ELEMS[case["c"]]), "flops": sites * (rows_out + rebuild)}
    if kind == "matvec":
        return {"bytes": sites * 8 * real * 12, "flops": sites * 288}
    if kind == "convert":
        return {"bytes": 2 * sites * (576 + 8 * real * ELEMS[case["a"]]), "flops": 0}
    return {"bytes": sites * 8 * real * 18, "flops": sites * 864}


# Measured against `exact` over the ranges above, and about four times what was seen: six-term FP64
# sums 0.98e-16 (1.1e-16 with row 2 rebuilt), FP32-pair sums (two 24-bit halves) 4.9e-15, FP32 sums
# with an FP32 b 5.5e-8, one rounding of each output to 11 bits 2.1e-4 or to 8 bits 1.6e-3.
REL = {"f64": 5e-16, "f32pair": 2e-14, "f32": 2.5e-7, "f16": 8e-4, "bf16": 7e-3}


def tolerance(case):
    if case["kind"] == "batch":
        return {"rel": REL["f32"]}  # half of the outputs are FP32
    if case["kind"] == "convert":
        return "exact" if case["a"] == "full" else {"rel": REL["f64"]}  # one rounding, or row 2 rebuilt
    return {"rel": REL["f32pair" if case["arith"] == "f32pair" else case["dtype"]]}


# ---- the products in 64 bits, with compensated sums, so that FP64 results can be judged -------------

def _split(x):
    t = x * 134217729.0  # 2^27 + 1: Veltkamp's splitting
    hi = t - (t - x)
    return hi, x - hi


def _dot(xs, ys):
    """sum_t xs[t] * ys[t] with error-free products and sums (Ogita, Rump and Oishi's Dot2)."""
    s = e = None
    for x, y in zip(xs, ys):
        p = x * y
        xh, xl = _split(x)
        yh, yl = _split(y)
        r = ((xh * yh - p) + xh * yl + xl * yh) + xl * yl
        if s is None:
            s, e = p, r
            continue
        t = s + p
        z = t - s
        e = e + (r + ((s - (t - z)) + (p - z)))
        s = t
    return s + e


def _product(a, b):
    """a [sites, 4, 3, 3, 2] x b [4, 3, n, 2], as [sites, 4, 3, n, 2]."""
    out = []
    for l in range(b.shape[2]):
        ar = [a[..., m, 0] for m in range(3)]
        ai = [a[..., m, 1] for m in range(3)]
        br = [b[:, m, l, 0].view(1, 4, 1) for m in range(3)]
        bi = [b[:, m, l, 1].view(1, 4, 1) for m in range(3)]
        re = _dot(ar + ai, br + [-x for x in bi])
        im = _dot(ar + ai, bi + br)
        out.append(torch.stack([re, im], -1))
    return torch.stack(out, -2)


def _row2(a):
    """Links [n, 6, 2] with row 2 = conj(row 0 x row 1) added: [n, 9, 2]."""
    u, v = a[:, :3], a[:, 3:]
    rows = []
    for k in range(3):
        p, q = (k + 1) % 3, (k + 2) % 3
        up, uq, vp, vq = u[:, p], u[:, q], v[:, p], v[:, q]
        re = _dot([up[:, 0], up[:, 1], uq[:, 0], uq[:, 1]], [vq[:, 0], -vq[:, 1], -vp[:, 0], vp[:, 1]])
        im = _dot([up[:, 0], up[:, 1], uq[:, 0], uq[:, 1]], [-vq[:, 1], -vq[:, 0], vp[:, 1], vp[:, 0]])
        rows.append(torch.stack([re, im], -1))
    return torch.cat([a, torch.stack(rows, 1)], 1)


def _links_product(a, b, rows, adjoint=False):
    """Links a [4 * sites, elements, 2] times b [4, 3, n, 2]: [4 * sites, rows * n, 2]."""
    n = b.shape[2]
    out = torch.empty(a.shape[0], rows * n, 2, dtype=torch.float64, device=a.device)
    for i in range(0, a.shape[0], CHUNK):
        x = a[i:i + CHUNK].to(torch.float64)
        if x.shape[1] == 6 and rows == 3:
            x = _row2(x)
        m = x.shape[0]
        x = x.reshape(m // 4, 4, x.shape[1] // 3, 3, 2)
        if adjoint:
            x = x.transpose(2, 3) * torch.tensor([1.0, -1.0], dtype=torch.float64, device=x.device)
        out[i:i + m] = _product(x, b).reshape(m, rows * n, 2)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        outs = {}
        for k, (sites, dtype) in enumerate(_batch_lattices(case)):
            a, b = _links(seed, sites, k)
            b = torch.from_numpy(b).cuda().view(4, 3, 3, 2)
            outs.setdefault(dtype, []).append(_links_product(a.to(TORCH[dtype]).view(-1, 9, 2), b, 3).view(-1))
        return [torch.cat(outs[t]) for t in ("f64", "f32") if t in outs]
    sites, dtype = case["sites"], TORCH[case["dtype"]]
    a, b = _links(seed, sites)
    bt = torch.from_numpy(b).cuda().view(4, 3, 3, 2)
    if kind == "convert":
        # the links themselves: what the form and the way back hold but for their rounding
        links = a.view(-1, 9, 2)
        form = _to_layout(links[:, :ELEMS[case["a"]]], case["layout"], torch.float64, sites, 0)
        return [form, links.reshape(-1)]
    a = a.to(dtype).view(-1, 9, 2)
    if kind == "matvec":
        v = bt[:, 0].reshape(4, 3, 1, 2)
        return _links_product(a, v, 3, adjoint=case["adjoint"]).view(-1)
    if kind == "host":
        return _links_product(a, bt, 3).view(-1).cpu()
    if case["op"] == "na":
        bt = (bt * torch.tensor([1.0, -1.0], dtype=torch.float64, device="cuda")).transpose(1, 2)
    rows = 3 if case["c"] == "full" else 2
    c = _links_product(a[:, :ELEMS[case["a"]]], bt, rows, adjoint=case["op"] == "an")
    return _to_layout(c, case["layout"], torch.float64, sites, case["stride"] * 8 // REAL[case["dtype"]])

"""The FP64 product's fixed-point rows (NATIVE arithmetic) against extended precision, at the edges of
their range: rows whose reals differ in size just inside and outside what the fixed-point form takes,
zeros, extreme and non-finite values, outputs whose terms are all small, and b matrices that suit it or
do not.

Bound. Every output real, fixed point or FP64 FMAs: six roundings, 6 * 2^-53 * sum |a||b| over its own
six terms. (In fixed point it is one rounding and 3.7 units of 2^-58 of full scale, where sum |a||b| is
at least 1/16 of full scale: 2.9 * 2^-53 * sum |a||b|.) Products that six FMAs give exactly are exact.
"""
import numpy as np
import pytest

import paper_2103_00571_gb300 as su3
import su3_inputs as gen

from gpu_helpers import run_form

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def links(a, n=9):
    """[V*72] doubles as complex extended precision [links, 3, 3]."""
    x = np.asarray(a, dtype=np.longdouble).reshape(-1, 3, 3, 2)
    return x[..., 0], x[..., 1]


def exact_and_bound(a, b):
    """c = a x b in extended precision and the per-real error bound, both [V*72]."""
    ar, ai = links(a)
    br, bi = (np.tile(x, (ar.shape[0] // 4, 1, 1)) for x in links(b))
    cr = np.einsum("qkm,qml->qkl", ar, br) - np.einsum("qkm,qml->qkl", ai, bi)
    ci = np.einsum("qkm,qml->qkl", ar, bi) + np.einsum("qkm,qml->qkl", ai, br)
    mag = lambda x, y, z, w: np.einsum("qkm,qml->qkl", abs(x), abs(y)) + np.einsum("qkm,qml->qkl", abs(z), abs(w))  # noqa: E731
    s = np.stack([mag(ar, br, ai, bi), mag(ar, bi, ai, br)], -1)
    return np.stack([cr, ci], -1).reshape(-1), (6 * U * s).reshape(-1)


def family(name, V, rng):
    a, b = gen.sites(7, 3, V), gen.bmat(7, 3, V)
    if name == "graded":  # the reals of a row spread over up to 2^9: on both sides of the limit
        a = a * 2.0 ** -rng.integers(0, 10, a.size)
    elif name == "spread":  # two reals of every row 2^-7 or 2^-8, the others near the largest
        a = np.sign(a) * rng.uniform(1, 2, a.size)
        for r in a.reshape(-1, 6):
            r[rng.permutation(6)[:3]] *= 2.0 ** -rng.integers(6, 10)
    elif name == "identity":  # links near the identity
        a = 1e-5 * a
        a.reshape(-1, 3, 3, 2)[:, range(3), range(3), 0] += 1.0
    elif name == "real":  # zero imaginary parts
        a.reshape(-1, 2)[:, 1] = 0.0
    elif name == "large":
        a = a * 2.0 ** 900
    elif name == "small":
        a = a * 2.0 ** -900
    elif name == "scaled":  # rows of sizes through the whole range of the fixed-point form
        a = (a.reshape(-1, 6) * 2.0 ** rng.integers(-720, 670, (a.size // 6, 1))).reshape(-1)
    elif name == "dyadic":  # low limbs of all ones and all zeros, exact powers of two
        a = np.sign(a) * np.where(rng.random(a.size) < 0.5, 1.0 - 2.0 ** -rng.integers(1, 54, a.size),
                                  2.0 ** -rng.integers(0, 4, a.size).astype(float))
    elif name == "small_terms":  # rows and columns whose large reals meet the small ones: sums of 2^-13
        a = np.sign(a) * rng.uniform(1, 2, a.size)
        a.reshape(-1, 3, 2)[:, 2, 0] *= 2.0 ** -2
        a.reshape(-1, 3, 2)[:, :, 1] *= 2.0 ** -8
        b = np.sign(b) * rng.uniform(1, 2, 72)
        b.reshape(4, 3, 3, 2)[:, :, 0] *= [0.0, 2.0 ** -4]
    elif name == "wide":  # reals of a row spread over up to 2^31, the limit of the form, and beyond
        a = a * 2.0 ** -rng.integers(0, 34, a.size)
    elif name == "smooth":  # links at various distances from the identity
        a = a * np.repeat(2.0 ** -rng.integers(1, 12, V * 4), 18)
        a.reshape(-1, 3, 3, 2)[:, range(3), range(3), 0] += 1.0
    elif name == "one_direction":  # b = 1 links beside random ones in every warp
        a.reshape(-1, 4, 18)[:, 0] = 0.0
        a.reshape(-1, 4, 3, 3, 2)[:, 0, range(3), range(3), 0] = 1.0
    elif name == "b_small":  # reals of b far below the largest of their matrix
        b = b * 2.0 ** -rng.permutation(np.repeat(np.arange(0, 36, 6), 12))
    elif name == "b_identity":
        b = np.zeros(72)
        b.reshape(4, 3, 3, 2)[:, range(3), range(3), 0] = 1.0
    elif name == "b_one_sparse":  # one matrix does not suit the form: all take FMAs
        b = b.copy()
        b.reshape(4, 3, 3, 2)[2, :, 1] = [[1e-3, 0], [1.0, 0], [0, 1e-4]]
    elif name == "b_scaled":
        b = b * np.repeat([2.0 ** 90, 1.0, 2.0 ** -60, 3.0], 18)
    return a, b


FAMILIES = ["random", "graded", "spread", "identity", "real", "large", "small", "scaled", "dyadic", "small_terms",
            "wide", "smooth", "one_direction", "b_small", "b_identity", "b_one_sparse", "b_scaled"]


@pytest.mark.parametrize("name", FAMILIES)
def test_error_bound(name):
    V = 1537
    a, b = family(name, V, np.random.default_rng(11))
    h = su3.Handle(0)
    c = run_form(h, a, b, su3.F64)
    want, bound = exact_and_bound(a, b)
    err = np.abs(c.astype(np.longdouble) - want)
    assert np.all(np.isfinite(c))
    assert np.all(err <= bound + 2.0 ** -1073), name
    if name in ("random", "b_scaled"):  # fixed point is the more exact: rows of FMAs throughout measure 9.8e-17
        assert np.linalg.norm(err.astype(float)) < 7e-17 * np.linalg.norm(want.astype(float))
    h.close()


def integers(shape, bits, rng):
    return rng.integers(1, 2 ** bits, shape) * rng.choice([-1.0, 1.0], shape)


@pytest.mark.parametrize("bits_a,bits_b", [(3, 3), (10, 10), (24, 24), (30, 3), (3, 30), (29, 20)])
def test_integers_are_exact(bits_a, bits_b):
    """Integer matrices whose products and sums FP64 holds come out exactly, as FP64 FMAs give them."""
    import torch
    V, rng = 1537, np.random.default_rng(5)
    a, b = integers(V * 72, bits_a, rng), integers(72, bits_b, rng)
    h = su3.Handle(0)
    want = exact_and_bound(a, b)[0].astype(np.float64)
    assert np.array_equal(run_form(h, a, b, su3.F64), want)
    d, dev = su3.Desc(su3.F64, su3.FULL18, su3.AOS, V), torch.from_numpy(a).cuda()
    at = np.ascontiguousarray(a.reshape(-1, 3, 3, 2).transpose(0, 2, 1, 3) * [1.0, -1.0]).reshape(-1)
    out, w = torch.empty_like(dev), torch.empty(V * 24, dtype=torch.float64, device="cuda")
    h.mult_op(su3.OP_AN, d, dev, b, d, out)
    h.mat_vec(d, dev, b.reshape(4, 3, 3, 2)[:, :, 0].copy(), w)
    h.sync()
    assert np.array_equal(out.cpu().numpy(), exact_and_bound(at, b)[0].astype(np.float64))
    assert np.array_equal(w.cpu().numpy(), want.reshape(-1, 3, 3, 2)[:, :, 0].reshape(-1))
    h.close()


@pytest.mark.parametrize("name", ["graded", "smooth", "one_direction", "wide"])
def test_rows_do_not_depend_on_their_warp(name):
    """Rows in fixed point, by FMAs and in part by each share warps: the same bits in any company."""
    V, rng = 1537, np.random.default_rng(13)
    a, b = family(name, V, rng)
    h = su3.Handle(0)
    c = run_form(h, a, b, su3.F64).reshape(V, 4, 18)
    for j in range(4):  # another order of the sites, and the direction's links alone (others zero)
        order = rng.permutation(V)
        alone = np.zeros((V, 4, 18))
        alone[:, j] = a.reshape(V, 4, 18)[order, j]
        assert np.array_equal(run_form(h, alone.reshape(-1), b, su3.F64).reshape(V, 4, 18)[:, j], c[order, j])
    h.close()


def test_non_finite_rows_stay_local():
    """Infinities and NaN give what FP64 arithmetic gives in their rows and touch no other row."""
    V = 70
    a, b = gen.sites(7, 4, V), gen.bmat(7, 4, V)
    bad = a.copy()
    bad[[5, 6 * 100 + 1, 6 * 333, 6 * 500 + 3]] = [np.inf, -np.inf, np.nan, 1.7e308]
    h = su3.Handle(0)
    c, good = run_form(h, bad, b, su3.F64), run_form(h, a, b, su3.F64)
    rows = np.zeros(V * 12, bool)
    rows[[0, 100, 333, 500]] = True
    assert np.array_equal(c.reshape(-1, 6)[~rows], good.reshape(-1, 6)[~rows])
    assert not np.isfinite(c.reshape(-1, 6)[[0, 100, 333]]).any()
    h.close()


@pytest.mark.parametrize("layout", [su3.AOS, su3.AOSOA32, su3.SOA])
@pytest.mark.parametrize("ri,ro", [(su3.FULL18, su3.FULL18), (su3.TWOROW12, su3.TWOROW12), (su3.TWOROW12, su3.FULL18)])
def test_rows_in_every_layout(layout, ri, ro):
    """The same rows to the same bits whatever the layout and the threads per link; ragged sizes."""
    h = su3.Handle(0)
    for V in (1, 9, 129, 1037):
        a, b = gen.sites(7, 5, V), gen.bmat(7, 5, V)
        a[: min(a.size, 900)] *= 2.0 ** -np.random.default_rng(V).integers(0, 12, min(a.size, 900))  # both kinds of row
        base = run_form(h, a, b, su3.F64, ri, ro)
        for tpl in (1, 3):
            got = run_form(h, a, b, su3.F64, ri, ro, layout=layout,
                           cfg=dict(block=128, tile_sites=32, stages=3, threads_per_link=tpl))
            assert np.array_equal(got, base), (V, tpl)
    h.close()


@pytest.mark.parametrize("name", ["random", "graded", "real", "dyadic", "small_terms", "wide", "b_small", "b_identity"])
def test_adjacent_products(name):
    """a^dagger b, a v and a^dagger v: the same bounds, with a's columns (conjugated) as rows."""
    import torch
    V = 777
    a, b = family(name, V, np.random.default_rng(12))
    h = su3.Handle(0)
    d = su3.Desc(su3.F64, su3.FULL18, su3.AOS, V)
    at = a.reshape(-1, 3, 3, 2).transpose(0, 2, 1, 3) * [1.0, -1.0]
    dev = torch.from_numpy(a).cuda()
    out = torch.empty_like(dev)
    h.mult_op(su3.OP_AN, d, dev, b, d, out)
    h.sync()
    want, bound = exact_and_bound(at.reshape(-1), b)
    assert np.all(np.abs(out.cpu().numpy().astype(np.longdouble) - want) <= bound)
    v = b.reshape(4, 3, 3, 2)[:, :, 0].copy()  # the first column of each matrix
    for adjoint, rows in ((False, a), (True, at)):
        want, _ = exact_and_bound(np.ascontiguousarray(rows).reshape(-1), b)
        bv = np.zeros((4, 3, 3, 2))
        bv[:, :, 0] = v
        _, bound = exact_and_bound(np.ascontiguousarray(rows).reshape(-1), bv.reshape(-1))
        w = torch.zeros(V * 24, dtype=torch.float64, device="cuda")
        h.mat_vec(d, dev, v, w, adjoint=adjoint)
        h.sync()
        pick = lambda x: x.reshape(-1, 3, 3, 2)[:, :, 0].reshape(-1)  # noqa: E731
        err = np.abs(w.cpu().numpy().astype(np.longdouble) - pick(want))
        assert np.all(err <= pick(bound)), (name, adjoint)
    h.close()


@pytest.mark.parametrize("tpl", [1, 3])
def test_batched_families(tpl):
    """Lattices whose b suits the form, does not, or has far exponents side by side in one batch: the bits
    of the single-lattice kernel from every entry point."""
    import ctypes
    import torch
    h, rng = su3.Handle(0), np.random.default_rng(17)
    items, keep = [], []
    for k, name in enumerate(FAMILIES):
        V = 129 + 16 * k
        a, b = family(name, V, rng)
        dev = torch.from_numpy(a).cuda()
        d = su3.Desc(su3.F64, su3.FULL18, su3.AOS, V)
        c = torch.zeros_like(dev)
        items.append(su3.BatchItem(d, dev.data_ptr(), c.data_ptr(), (ctypes.c_double * 72)(*b)))
        keep.append((name, dev, c, run_form(h, a, b, su3.F64)))
    h.set_batched_cfg(block=128 if tpl == 3 else 64, tile_sites=32, stages=3, ctas_per_sm=4, threads_per_link=tpl)
    calls = [lambda: h.mult_batched(items, use_graph=False), lambda: h.mult_batched(items, use_graph=True),
             lambda: h.mult_batched(items, use_graph=True)]
    if tpl == 1:  # the static entry point has the default shape
        arr, stream = (su3.BatchItem * len(items))(*items), torch.cuda.current_stream().cuda_stream
        calls.append(lambda: su3.lib().su3_mult_batched_static(len(items), arr, ctypes.c_void_p(stream)))
    for call in calls:
        for _, _, c, _ in keep:
            c.zero_()
        call()
        h.sync()
        torch.cuda.synchronize()
        for name, _, c, want in keep:
            assert np.array_equal(c.cpu().numpy(), want), name
    h.close()

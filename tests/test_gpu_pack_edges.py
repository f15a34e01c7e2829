"""su3_pack and su3_unpack at the edges of their rounding and of their tiles: ties and values next to
them, the ends of each type's range, zeros, subnormals, infinities and NaN, and ragged last tiles."""
import numpy as np
import pytest

import oracle
import paper_2103_00571_gb300 as su3

pytestmark = pytest.mark.gpu

ROUND = {su3.F32: lambda x: oracle.round_float(x).astype(np.float64),
         su3.F16: lambda x: oracle.widen_half(oracle.round_half(x)),
         su3.BF16: lambda x: oracle.widen_bf16(oracle.round_bf16(x))}


def values():
    """Doubles at and beside the rounding boundaries of 8, 11 and 24 bits through every size."""
    out = [0.0, -0.0, np.inf, -np.inf, 5e-324, 1e-310, 2.0 ** -149, 2.0 ** -150, 65504.0, 65519.999, 65520.0, 1e300]
    for e in (-150, -149, -133, -127, -126, -125, -25, -24, -15, -14, -1, 0, 1, 15, 16, 126, 127, 128, 900):
        for bits in (8, 11, 24):
            for m in (1.0, 1.0 + 2.0 ** (1 - bits), 2.0 - 2.0 ** (1 - bits)):
                tie = (m + 2.0 ** -bits) * 2.0 ** e
                out += [tie, np.nextafter(tie, 0), np.nextafter(tie, np.inf), m * 2.0 ** e]
    x = np.array(out)
    return np.concatenate([x, -x])


@pytest.mark.parametrize("layout", [su3.AOS, su3.AOSOA32, su3.SOA])
@pytest.mark.parametrize("dtype", [su3.F32, su3.F16, su3.BF16])
def test_rounds_once(dtype, layout):
    import torch
    h = su3.Handle(0)
    x = values()
    for V in (1, 31, 32, 33, 65):
        a = np.resize(np.roll(x, 7 * V), V * 72)
        d = su3.Desc(dtype, su3.FULL18, layout, V)
        buf = torch.zeros(su3.array_bytes(d), dtype=torch.uint8, device="cuda")
        back = torch.empty(V * 72, dtype=torch.float64, device="cuda")
        h.pack(torch.from_numpy(a).cuda(), d, buf)
        h.unpack(d, buf, back)
        h.sync()
        got, want = back.cpu().numpy(), ROUND[dtype](a)
        assert np.array_equal(got.view(np.uint64), want.view(np.uint64)), V
    h.close()


@pytest.mark.parametrize("layout", [su3.AOS, su3.AOSOA32, su3.SOA])
@pytest.mark.parametrize("dtype", [su3.F64, su3.F32, su3.F16, su3.BF16])
def test_two_row_and_nan(dtype, layout):
    """Two-row forms drop row 2 and rebuild it in FP64; a NaN stays in its own link."""
    import torch
    h = su3.Handle(0)
    rng = np.random.default_rng(3)
    for V in (1, 33, 64):
        a = rng.standard_normal(V * 72)
        d = su3.Desc(dtype, su3.TWOROW12, layout, V)
        buf = torch.zeros(su3.array_bytes(d), dtype=torch.uint8, device="cuda")
        back = torch.empty(V * 72, dtype=torch.float64, device="cuda")
        bad = a.copy()
        bad[18 * (4 * V - 1)] = np.nan
        for src in (a, bad):
            h.pack(torch.from_numpy(src).cuda(), d, buf)
            h.unpack(d, buf, back)
            h.sync()
            got = back.cpu().numpy().reshape(-1, 18)
            n = got.shape[0] - (src is bad)
            rows = src.reshape(-1, 18)[:n, :12]
            rows = rows if dtype == su3.F64 else ROUND[dtype](np.ascontiguousarray(rows).reshape(-1)).reshape(-1, 12)
            assert np.array_equal(got[:n, :12], rows)
            want = oracle.tworow_expand(np.ascontiguousarray(rows)).reshape(-1, 18)
            assert np.allclose(got[:n], want, rtol=0, atol=4 * 2.0 ** -52 * 32)  # four products of up to ~6^2
        assert np.isnan(got[-1]).any()
    h.close()

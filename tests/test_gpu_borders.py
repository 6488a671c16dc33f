"""Image borders by mirrored data, unaligned bands, and where work items start.

Sizes at the edges of strips (a strip whose last column, or whose halo, lies
outside the image), widths shorter than a halo, odd and even, in both tile
widths, forward and inverse, against the FP64 oracle; segments of every short
length; the row decomposition of batches.
"""
import numpy as np
import pytest
import torch

from oracle import lifting as L
from paper_1705_08266_gb300 import dwt2d as D
from tests.parity_util import (assert_forward_matches, assert_inverse_matches, device_image, host,
                               make_input)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    D.lib()


# strips store 104 / 120 columns (2 / 1 fused levels) with 2 columns per lane
# and 224 / 240 with 4
EDGE_WIDTHS = [2, 3, 4, 5, 6, 7, 9, 12, 15, 16, 17, 18, 31, 33, 103, 104, 105, 106, 113, 119, 120, 121, 122,
               207, 208, 209, 210, 223, 224, 225, 226, 239, 240, 241, 242, 447, 448, 449, 450]


@pytest.mark.parametrize("cols", [2, 4])
@pytest.mark.parametrize("wavelet,scheme", [("cdf97", "nonsep_reduced"), ("cdf97", "separable"),
                                            ("cdf97", "nonsep"), ("legall53", "nonsep_reduced")])
def test_strip_edges(wavelet, scheme, cols):
    for w in EDGE_WIDTHS:
        for h, levels in ((19, 3), (40, 2), (2, 1)):
            x = make_input(wavelet, h, w, seed=w * 3 + h)
            plan = D.Plan(h, w, levels, wavelet, scheme,
                          options=dict(fwd_cols_per_lane=cols, inv_cols_per_lane=cols))
            ws = plan.workspace()
            tag = f"{wavelet} {scheme} cols={cols} {h}x{w} L{levels}"
            c = plan.forward(device_image(x), workspace=ws)
            assert_forward_matches(host(c), x, levels, wavelet, tag)
            ref = L.forward(x, levels, wavelet).astype(x.dtype)
            y = plan.inverse(device_image(ref), workspace=ws)
            assert_inverse_matches(host(y), ref, levels, wavelet, x, tag)
            assert plan.status(ws) == 0, tag


# rows that leave 1 .. a slot's rows in the last segment, at both fusion depths
@pytest.mark.parametrize("wavelet", ["cdf97", "legall53"])
@pytest.mark.parametrize("fuse", [1, 2])
def test_slot_starts(wavelet, fuse):
    """Work items start at any row (one fused level) or pair of rows (two):
    every segment length from 1 up gives the same bits, forward and inverse."""
    for h in (37, 38, 39, 40, 130):
        w = 150
        x = make_input(wavelet, h, w, seed=h)
        xd = device_image(x)
        ref = None
        for seg in (1, 2, 3, 4, 5, 7, 8, 1000, 0):
            opts = dict(fuse_max=fuse)
            if seg:
                opts.update(min_segment=seg, fwd_warps_per_sm=60000, inv_warps_per_sm=60000)
            plan = D.Plan(h, w, 3, wavelet, options=opts)
            ws = plan.workspace()
            c = plan.forward(xd, workspace=ws)
            y = plan.inverse(c, workspace=ws)
            torch.cuda.synchronize()
            assert plan.status(ws) == 0
            if ref is None:
                ref = (c.clone(), y.clone())
                assert_forward_matches(host(c), x, 3, wavelet, f"{h} fuse {fuse}")
            assert torch.equal(c, ref[0]) and torch.equal(y, ref[1]), (h, fuse, seg)


def test_default_batch_rows_equal_tuned_ones():
    """The default row decomposition of batches (by the size of each launch,
    4 columns per lane for large ones) gives the bits of a fixed one."""
    rng = np.random.default_rng(5)
    jobs = []
    for _ in range(24):
        h, w = int(rng.integers(65, 3000)), int(rng.integers(65, 3000))
        x = D.empty_image(h, w)
        x.copy_(torch.rand(h, w, device="cuda"))
        jobs.append((x, D.empty_image(h, w), int(rng.integers(1, 6)), "cdf97", 0))
    outs = []
    for tuning in (None, dict(warps_per_sm=24, cols_per_lane=2)):
        b = D.Batch(jobs, tuning=tuning)
        ws = b.workspace()
        b.upload(ws)
        b.launch(ws)
        torch.cuda.synchronize()
        assert b.status(ws) == 0
        outs.append([d.clone() for _s, d, _l, _w, _i in jobs])
    for a, c in zip(*outs):
        assert torch.equal(a, c)


@pytest.mark.parametrize("dtype", [torch.float32, torch.int32, torch.float16])
@pytest.mark.parametrize("h,w,levels", [(2500, 5000, 2), (3001, 4097, 1), (6000, 1500, 3), (3000, 9000, 2),
                                        (9999, 10001, 2)])
def test_middle_sizes_equal_one_wave(h, w, levels, dtype):
    """Between the small launches and the large ones the wave count follows the
    segments' length: the default plan gives the bits of one-wave launches."""
    wavelet = "legall53" if dtype == torch.int32 else "cdf97"
    x = D.empty_image(h, w, dtype)
    x.copy_((torch.rand(h, w, device="cuda") * 100).to(dtype))
    outs = []
    for options in (None, dict(fwd_warps_per_sm_large=-1, inv_warps_per_sm_large=-1)):
        plan = D.Plan(h, w, levels, wavelet, "nonsep_reduced", dtype, options=options)
        ws = plan.workspace()
        c = plan.forward(x, workspace=ws)
        y = plan.inverse(x, workspace=ws)
        torch.cuda.synchronize()
        assert plan.status(ws) == 0
        outs.append((c, y))
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])


@pytest.mark.parametrize("h,w,levels", [(513, 512, 3), (1080, 1920, 5), (1601, 2499, 4), (2048, 2049, 6),
                                        (2700, 5001, 5)])
@pytest.mark.parametrize("scheme", ["nonsep_reduced", "separable"])
def test_single_level_launches_equal_fused_ones(h, w, levels, scheme):
    """Small float32 levels have forward launches of their own: the same bits
    as fused pairs, and an inverse that takes its own groups."""
    x = D.empty_image(h, w)
    x.copy_(torch.rand(h, w, device="cuda") * 255)
    outs = []
    for options in (None, dict(fuse_first=2, fuse_max=2)):
        plan = D.Plan(h, w, levels, "cdf97", scheme, options=options)
        ws = plan.workspace()
        c = plan.forward(x, workspace=ws)
        y = plan.inverse(c, workspace=ws)
        torch.cuda.synchronize()
        assert plan.status(ws) == 0
        fwd, inv = plan.launch_info(), plan.launch_info(inverse=True)
        assert sum(f for f, _q, _w in fwd) == levels and sum(f for f, _q, _w in inv) == levels
        outs.append((c, y))
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16])
@pytest.mark.parametrize("scheme", ["nonsep_reduced", "separable", "nonsep"])
def test_nonfinite_coefficients_stay_where_they_belong(scheme, dtype):
    """Levels one column wide have no HL and HH bands, and the columns beside
    their LL hold another level's details: an infinity or a NaN there may only
    reach the samples that the oracle's inverse makes non-finite.  Wider images
    likewise, where a box holds a neighbouring band past the border."""
    rng = np.random.default_rng(17)
    for h, w in [(40, 1), (1, 40), (40, 2), (64, 3), (33, 5), (64, 8), (7, 300), (37, 241)]:
        for levels in (1, 2, 3, 6):
            for options in (None, dict(fuse_max=1), dict(inv_cols_per_lane=4)):
                plan = D.Plan(h, w, levels, "cdf97", scheme, dtype, options=options)
                ws = plan.workspace()
                for k in range(6):
                    r, c = int(rng.integers(0, h)), min(k, w - 1) if k < 3 else int(rng.integers(0, w))
                    x = np.full((h, w), 0.5)
                    x[r, c] = (np.inf, np.nan)[k % 2]
                    with np.errstate(invalid="ignore"):
                        ref = L.inverse(x, levels, "cdf97")
                    xd = D.empty_image(h, w, dtype)
                    xd.copy_(torch.from_numpy(x))
                    y = host(plan.inverse(xd, workspace=ws)).astype(np.float64)
                    bad = np.isfinite(ref) & ~np.isfinite(y)
                    assert not bad.any(), (h, w, levels, options, r, c, np.argwhere(bad)[:4].tolist())


def test_default_columns_of_a_large_batch_equal_two():
    """A float32 batch large enough for 4 columns per lane by default gives the
    bits of 2 columns per lane."""
    x = D.empty_image(8192, 8192)
    x.copy_(torch.rand(8192, 8192, device="cuda"))
    outs, warps = [], []
    for tuning in (None, dict(cols_per_lane=2)):
        jobs = [(x, D.empty_image(8192, 8192), 3, "cdf97", 0) for _ in range(6)]
        b = D.Batch(jobs, tuning=tuning)
        ws = b.workspace()
        b.upload(ws)
        b.launch(ws)
        torch.cuda.synchronize()
        assert b.status(ws) == 0
        outs.append([d for _s, d, _l, _w, _i in jobs])
        warps.append(b.info()[1])
    assert warps[0] != warps[1]
    for a, c in zip(*outs):
        assert torch.equal(a, c)


@pytest.mark.parametrize("scheme", ["nonsep_reduced", "separable", "nonsep"])
def test_nonfinite_pixels_stay_where_they_belong(scheme):
    """Forward, up to three fused levels: an infinity or a NaN of the image only
    reaches the coefficients that the oracle makes non-finite, also where a
    level is one row or one column."""
    rng = np.random.default_rng(19)
    for h, w in [(1, 40), (2, 40), (3, 64), (40, 2), (64, 3), (5, 33), (7, 300), (37, 241)]:
        for levels in (1, 2, 3, 6):
            for options in (None, dict(fuse_max=1), dict(fwd_cols_per_lane=4), dict(fuse_first=3, fuse_max=3)):
                plan = D.Plan(h, w, levels, "cdf97", scheme, options=options)
                ws = plan.workspace()
                for k in range(6):
                    r, c = int(rng.integers(0, h)), int(rng.integers(0, w))
                    x = np.full((h, w), 0.5)
                    x[r, c] = (np.inf, np.nan)[k % 2]
                    with np.errstate(invalid="ignore"):
                        ref = L.forward(x, levels, "cdf97")
                    xd = D.empty_image(h, w)
                    xd.copy_(torch.from_numpy(x))
                    y = host(plan.forward(xd, workspace=ws))
                    bad = np.isfinite(ref) & ~np.isfinite(y)
                    assert not bad.any(), (h, w, levels, options, r, c, np.argwhere(bad)[:4].tolist())


# 16-bit strips start on 8 elements: 96 / 112 columns (2 / 1 fused levels) with
# 2 columns per lane, 224 / 240 with 4.  Tolerances of 16-bit storage: a stored
# value's rounding times the largest gain it passes through.
TOL_16 = {torch.float16: 2e-3, torch.bfloat16: 1.6e-2}


@pytest.mark.parametrize("cols", [2, 4])
@pytest.mark.parametrize("scheme", ["nonsep_reduced", "separable", "nonsep"])
@pytest.mark.parametrize("dtype", list(TOL_16))
def test_strip_edges_of_16bit_storage(dtype, scheme, cols):
    for w in [2, 3, 5, 8, 9, 17, 95, 96, 97, 98, 111, 112, 113, 114, 191, 192, 193, 194, 223, 224, 225, 226,
              239, 240, 241]:
        for h, levels in ((19, 3), (2, 1)):
            x = make_input("cdf97", h, w, seed=w * 3 + h)
            xq = torch.from_numpy(x / float(np.max(np.abs(x)))).to(dtype)
            plan = D.Plan(h, w, levels, "cdf97", scheme, dtype,
                          options=dict(fwd_cols_per_lane=cols, inv_cols_per_lane=cols))
            ws = plan.workspace()
            src = D.empty_image(h, w, dtype)
            src.copy_(xq)
            ref = L.forward(xq.to(torch.float64).numpy(), levels, "cdf97")
            got = host(plan.forward(src, workspace=ws).to(torch.float64))
            assert float(np.max(np.abs(got - ref))) <= TOL_16[dtype], (h, w, levels)
            cq = torch.from_numpy(ref).to(dtype)
            src.copy_(cq)
            back = L.inverse(cq.to(torch.float64).numpy(), levels, "cdf97")
            got = host(plan.inverse(src, workspace=ws).to(torch.float64))
            assert float(np.max(np.abs(got - back))) <= TOL_16[dtype], (h, w, levels, "inverse")
            assert plan.status(ws) == 0


@pytest.mark.parametrize("wavelet,scheme", [("cdf97", "nonsep_reduced"), ("cdf97", "separable"),
                                            ("cdf97", "nonsep"), ("legall53", "nonsep_reduced")])
def test_strip_edges_of_three_fused_levels(wavelet, scheme):
    """Strips of 192 (CDF 9/7) and 224 (5/3) columns, whose halo is 28 and 14."""
    for w in EDGE_WIDTHS + [27, 28, 29, 57, 191, 192, 193, 194, 219, 220, 221, 383, 384, 385]:
        for h, levels in ((23, 3), (40, 5)):
            x = make_input(wavelet, h, w, seed=w * 5 + h)
            plan = D.Plan(h, w, levels, wavelet, scheme, options=dict(fuse_first=3, fuse_max=3))
            ws = plan.workspace()
            tag = f"{wavelet} {scheme} {h}x{w} L{levels}"
            assert_forward_matches(host(plan.forward(device_image(x), workspace=ws)), x, levels, wavelet, tag)
            ref = L.forward(x, levels, wavelet).astype(x.dtype)
            y = plan.inverse(device_image(ref), workspace=ws)
            assert_inverse_matches(host(y), ref, levels, wavelet, x, tag)
            assert plan.status(ws) == 0, tag

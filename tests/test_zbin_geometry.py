"""The z order of team cells on the CPU: float32 replays of the kernel's bin
formula.  Bins are monotone in z inside a cell, and a particle of the same or a
later bin is never more than the stated width below."""
import numpy as np
import pytest

from paper_2003_11468_gb300 import fof

F = np.float32


@pytest.mark.parametrize("box,l_over_h,nc", [(1.0, 0.2, 3), (100.0, 0.3, 1520), (50.0, 0.45, 351), (123.456, 0.3, 4096),
                                             (7.3e-4, 0.9, 17), (3.0e7, 0.25, 2048)])
def test_bins_monotone_and_width(box, l_over_h, nc):
    opt = fof.fof_options()
    opt.cells_per_axis = nc
    geo = fof.fof_box_geometry(box, l_over_h * box / nc, 1000, opt)
    nc = geo.cells_per_axis
    rng = np.random.default_rng(nc)
    cells = np.unique(np.concatenate([[0, nc - 1], rng.integers(0, nc, 40)]))
    inv_zb = F(32.0 * nc / box)
    width = F(np.nextafter(F(1.125 * box / (32.0 * nc)), F(np.inf)))
    for cz in cells:
        edges = (cz + np.arange(33) / 32.0) * (box / nc)
        z = np.concatenate([rng.uniform(edges[0], edges[-1], 400), edges, np.nextafter(edges, 0), np.nextafter(edges, box)])
        z = np.concatenate([F(z), np.nextafter(F(edges), F(0)), np.nextafter(F(edges), F(np.inf))])
        z = z[(z >= 0) & (z <= F(geo.xmax))]
        # members of the cell: the fine coordinate's quotient, as the kernels take it
        fine = np.clip((z * F(geo.inv_fine)).astype(np.int64), 0, geo.fine_per_axis - 1)
        z = np.sort(z[fine // geo.sub_cells == cz])
        bins = np.clip((z * inv_zb).astype(np.int64) - 32 * cz, 0, 31)
        assert np.all(np.diff(bins) >= 0)
        highest = np.array([z[bins == k].max() if np.any(bins == k) else F(0) for k in range(32)])
        lowest = np.array([z[bins >= k].min() if np.any(bins >= k) else F(np.inf) for k in range(32)])
        for k in range(32):
            if np.any(bins == k):
                assert F(highest[k] - width) <= lowest[k]


@pytest.mark.parametrize("t_hi", [0.0, 1.4e-45, 1.2e-38, 3.7e-9, 0.04, 1.0, 16384.0, 3.4028235e38])
def test_threshold_as_sign_of_a_difference(t_hi):
    """s2 <= t_hi and s2 < t as the sign bit of s2 minus a float32, the form the
    team kernel's packed pair tests take, on the neighbours of each threshold."""
    t = F(t_hi)
    with np.errstate(over="ignore"):
        above = (t.view(np.uint32) + np.uint32(1)).view(F)
        s2 = np.concatenate([t.view(np.uint32) + np.arange(-40, 40), [0, 1, 2, 0x00800000, 0x7f7fffff, 0x7f800000]])
        s2 = np.clip(s2, 0, 0x7f800000).astype(np.uint32).view(F)
        s2 = s2[~(np.isinf(s2) & np.isinf(above))]      # inf - inf: no sign on the device, and not <= t_hi
        assert np.array_equal(np.signbit(s2 - above), s2 <= t)
        assert np.array_equal(np.signbit(s2 - t), s2 < t)

"""Edges of the FP32 walker's plane arithmetic against the FP64 oracle: its two
forms (every source on the 1/16-cell lattice, or any position), sources on and
within rounding of cell planes and box faces, axes longer than the lattice
form takes, and both forms' optical depths up to the termination.

Counts per level and the created-set checksum must be bit-exact; k_ph, Gamma
and the budget within the bounds of tests/parity.py.
"""
import numpy as np
import pytest

import parity
from paper_1012_2865_gb300 import synth

pytestmark = pytest.mark.gpu

LATTICE = [(0.0, 0.0, 0.0), (8.0, 5.0, 3.0), (4.5, 7.5, 2.5), (3.0625, 9.9375, 6.5), (16.0, 11.0, 7.0)]
BESIDE = [(8.0 + 1e-12, 5.0 - 1e-9, 3.0 + 1e-7), (1e-13, 11.0 - 1e-9, 3.5), (16.0 - 1e-12, 5.5, 1e-9),
          (7.3, 5.000001, 2.9999999), (8.0, 5.0, 3.3)]


def _grid(dims, cells, xlo, seed=3):
    rng = np.random.default_rng(seed)
    box = synth.box_cm(dims[0], 6.6 * dims[0] / 32)
    dx = box / dims[0]
    n = len(cells)
    n_H = 2e-3 if dims == (1, 1, 1) else synth.lognormal_density(None, mean=2e-3, seed=seed, dims=dims)
    return synth._grid(dims, box, n_H,
                       rng.uniform(xlo, 1.0, int(np.prod(dims))) if xlo > 0 else 1e-4, np.asarray(cells) * dx,
                       np.full(n, 1e49), rng.uniform(13.6, 29.6, n), np.full(n, synth.SIGMA_HI))


@pytest.mark.parametrize("xlo", [0.9, 0.0])  # rays that are absorbed; rays that leave the box
@pytest.mark.parametrize("cells", [LATTICE, BESIDE, LATTICE + BESIDE], ids=["lattice", "beside", "both"])
def test_sources_on_and_beside_planes(cells, xlo):
    g = _grid((16, 11, 7), cells, xlo)
    _, b, r = parity.run_gpu(g, "fp32_mixed")
    parity.assert_trace_parity(g, b, r, parity.run_oracle(g), "fp32_mixed")


@pytest.mark.parametrize("dims,cells", [
    ((1, 1, 1), [(0.5, 0.5, 0.5), (0.1, 0.7, 0.9)]),
    ((5000, 2, 3), [(2500.5, 0.5, 1.5), (4096.5, 1.0, 2.0), (0.3, 1.9, 0.1)]),
    ((2, 4097, 1), [(1.0, 4096.5, 0.5), (0.25, 17.0, 0.5)]),
], ids=["one-cell", "5000", "4097"])
def test_short_and_long_axes(dims, cells):
    g = _grid(dims, cells, 0.0)
    _, b, r = parity.run_gpu(g, "fp32_mixed")
    parity.assert_trace_parity(g, b, r, parity.run_oracle(g), "fp32_mixed")


@pytest.mark.parametrize("seed", range(6))
def test_termination_after_a_clipped_dense_cell(seed):
    """A level-6 ray that clips 2e-10 cell lengths off a cell dense enough to
    take most of its optical depth there: what FP32 pairs know of that length
    (about 1e-12) leaves an error that only the bound its children inherit
    covers, and they terminate in thin gas, where it is cells wide."""
    import oracle
    rng = np.random.default_rng(seed)
    dims, dx = (48, 48, 48), 2.0 ** 60
    n = oracle.pix2vec(6, np.arange(4 ** 6))
    n = n[np.all((n > 0.45) & (n < 0.7), axis=1)]
    n = n[rng.integers(len(n))]
    s = rng.uniform(2.0, 4.0, 3)
    i = np.ceil(s[0] + 20.0 * n[0])
    t = (i - s[0]) / n[0]                      # between the splits at 13.8 and 27.7
    j = np.ceil(s[1] + t * n[1])
    s[1] = j - (t + 2e-10) * n[1]              # plane j follows plane i at once
    cell = int(i) + 48 * (int(j) - 1 + 48 * int(s[2] + t * n[2]))
    f_term, thin = 0.9, 1e-4
    depth = np.full(48 ** 3, thin)             # optical depth per cell length
    depth[cell] = (-np.log(f_term) - 37.0 * thin) / 2e-10
    g = synth._grid(dims, 48 * dx, depth / (synth.SIGMA_HI * dx), 1.0, [s * dx], [1e49], [20.0], [synth.SIGMA_HI])
    _, b, r = parity.run_gpu(g, "fp32_mixed", f_term=f_term)
    parity.assert_trace_parity(g, b, r, parity.run_oracle(g, f_term=f_term), "fp32_mixed", exact_segments=True)


def test_diagonal_ties_need_no_fallback():
    """Sources on the lattice in a launch that holds others too, and in the
    allocation-free trace: the ties of their 45-degree rays are exact there as
    well, so each source takes the FP64 fallbacks it takes by itself."""
    import torch
    from paper_1012_2865_gb300 import native
    dims, alone = (16, 11, 7), 0
    lattice = [(4.5, 7.5, 2.5), (8.5, 5.5, 3.5), (3.5, 2.5, 1.5), (3.0625, 9.9375, 6.5), (8.0, 5.0, 3.0)]
    for cells in (lattice, BESIDE):
        alone += parity.run_gpu(_grid(dims, cells, 0.0), "fp32_mixed")[1]["fallbacks"]
    _, b, _ = parity.run_gpu(_grid(dims, lattice + BESIDE, 0.0), "fp32_mixed")
    assert b["fallbacks"] == alone
    g = _grid(dims, lattice, 0.0)
    _, b, _ = parity.run_gpu(g, "fp32_mixed")
    dev = lambda a, t: torch.tensor(a, dtype=t, device="cuda")
    n = int(np.prod(dims))
    out = torch.zeros((2, n), dtype=torch.float32, device="cuda")
    na = native.rt_trace_noalloc(dims, g["box_len_cm"], dev(g["n_H"] * g["x_HI"], torch.float32),
                                 dev(g["n_H"], torch.float64), dev(g["x_HI"], torch.float64), out[0], out[1],
                                 g["pos_cm"], g["ndot"], g["e_ph_eV"], g["sigma_cm2"],
                                 native.trace_params(**synth.DEFAULT_PARAMS))
    assert na["fallbacks"] == b["fallbacks"]


def test_lengths_along_a_diagonal_in_the_general_form():
    """Unsplit rays through next to nothing: k_ph is the path length per cell,
    also along the 45-degree rays of lattice sources, whose ties the general
    form (an off-lattice source is there too) meets with two pairs for one
    distance.  An FP32 unit of a radius of 40 is 4e-6 cells."""
    dims, dx = (64, 64, 64), 2.0 ** 60
    rng = np.random.default_rng(5)
    cells = [(x + 0.5, y + 0.5, z + 0.5) for x, y, z in rng.integers(2, 20, (7, 3))] + [(50.3, 50.7, 3.1)]
    g = synth._grid(dims, 64 * dx, 1e-9 / (synth.SIGMA_HI * dx), 1.0, np.asarray(cells) * dx, np.full(8, 1e49),
                    np.full(8, 20.0), np.full(8, synth.SIGMA_HI))
    o = parity.run_oracle(g, level0=2, max_level=2)
    _, b, r = parity.run_gpu(g, "fp32_mixed", level0=2, max_level=2)
    np.testing.assert_array_equal(b["counts"], o["counts"])
    length = o["kph"][o["kph"] > 0].mean()
    np.testing.assert_allclose(r["kph"], o["kph"], rtol=1e-6, atol=1e-6 * length)


T3 = 16.0 / 3.0


@pytest.mark.parametrize("xlo", [0.9, 0.0])
@pytest.mark.parametrize("cells,exact", [
    ([(T3, T3, 2.1), (T3, T3, 6.9)], True), ([(8.3, 10.3, 3.3)], True), ([(8.3, 5.7, 3.3), (9.7, 4.3, 0.2)], False),
    ([(0.7, 0.3, 5.1)], True), ([(8.3, 8.7, 2.0)], True), ([(8.3, 4.3, 3.3), (1.0 / 3.0, 4.0 / 3.0, 3.0)], False),
    ([(8.3, 4.3 + 1e-13, 3.3), (9.7, 4.3 - 1e-14, 2.2)], False), ([(2.5, 9.25, 3.1), (2.5, 9.5, 3.1)], True)],
    ids=["thirds", "equal", "opposite", "opposite-exact", "opposite-exact-2", "rounded", "near", "lattice-xy"])
def test_ties_off_the_lattice(cells, exact, xlo):
    """45-degree rays of sources whose x and y lie equally far from planes: where
    that holds exactly the ties need no fallback, and where the positions'
    rounding sets the planes apart by 1e-16 to 1e-13, FP64 decides."""
    g = _grid((16, 11, 7), cells, xlo)
    _, b, r = parity.run_gpu(g, "fp32_mixed")
    parity.assert_trace_parity(g, b, r, parity.run_oracle(g), "fp32_mixed")
    s = np.asarray(g["pos_cm"]) / (g["box_len_cm"] / 16)  # as the library has them
    frac = s - np.rint(s)
    tied = (np.abs(frac[:, 0]) == np.abs(frac[:, 1])).all()
    if exact and tied:
        assert b["fallbacks"] == 0


def test_near_ties_of_many_packages():
    """Planes that nearly tie at every step, along each pair of axes, for
    packages of several levels and sources in one warp: the direction kept for
    such decisions is the package's own."""
    cells = [(5.3, 12.3, 3.3), (5.3 + 1e-14, 9.3, 2.7), (1.1, 8.1, 4.1), (8.1, 1.1 + 2e-15, 4.1), (2.7, 9.3, 4.7)]
    g = _grid((16, 16, 9), cells, 0.0)
    _, b, r = parity.run_gpu(g, "fp32_mixed", phi_c=3.0)
    parity.assert_trace_parity(g, b, r, parity.run_oracle(g, phi_c=3.0), "fp32_mixed")
    assert b["fallbacks"] > 500

"""State and rate fields through the C ABI at sizes where the kernels behind
them change form: odd cell counts and misaligned device arrays (no 16-byte
accesses), a rejected state that must leave the grid as it was, k_ph and Gamma
of a mixed grid written and read back in either type and place, and timestep
tiles that the grid does not fill."""
import numpy as np
import pytest

import parity
from oracle import timestep
from paper_1012_2865_gb300 import native, synth

pytestmark = pytest.mark.gpu


def _medium(dims, seed=4, sources=2):
    rng = np.random.default_rng(seed)
    box = synth.box_cm(dims[0], 6.6 * dims[0] / 32)
    n = int(np.prod(dims))
    pos, ndot, e, sg = synth.random_sources(dims, box / dims[0], sources, 1e48, 1e49, rng)
    return synth._grid(dims, box, rng.uniform(1e-3, 1e-2, n), rng.uniform(1e-3, 1.0, n), pos, ndot, e, sg)


@pytest.mark.parametrize("precision", ["fp64", "fp32_mixed"])
@pytest.mark.parametrize("dims,skip", [((3, 5, 7), 0), ((4, 5, 6), 0), ((4, 5, 6), 1), ((33, 9, 8), 1)])
def test_device_state_replaces_and_rejects(precision, dims, skip):
    import torch
    g = _medium(dims)
    n = int(np.prod(dims))
    rng = np.random.default_rng(8)
    want = _medium(dims, seed=9)
    want.update({k: g[k] for k in ("pos_cm", "ndot", "e_ph_eV", "sigma_cm2")})

    def dev(a):  # a contiguous device array, off 16-byte alignment where skip is 1
        t = torch.zeros(n + skip, dtype=torch.float64, device="cuda")
        t[skip:] = torch.tensor(a, dtype=torch.float64)
        return t[skip:]

    grid = native.Grid(parity.ctx(), g, precision)
    for field, cell, value in (("x_HI", n - 1, 1.5), ("x_HI", 0, float("nan")), ("n_H", n // 2, -1.0)):
        bad = {"x_HI": rng.uniform(0, 1, n), "n_H": rng.uniform(0, 1, n)}
        bad[field][cell] = value
        with pytest.raises(native.RtError, match=rf"{field}\[{cell}\]"):
            native.rt_set_state(grid.h, dev(bad["x_HI"]), n_H=dev(bad["n_H"]))
    np.testing.assert_array_equal(grid.rates()["x_HI"], g["x_HI"])
    ref = native.Grid(parity.ctx(), want, precision)
    native.rt_set_state(grid.h, dev(want["x_HI"]), dev(want["x_HII"]), dev(want["n_H"]))
    a, b = grid.trace(**synth.DEFAULT_PARAMS), ref.trace(**synth.DEFAULT_PARAMS)
    np.testing.assert_array_equal(a["counts"], b["counts"])
    assert a["segments"] == b["segments"]
    np.testing.assert_array_equal(grid.rates()["x_HI"], want["x_HI"])
    np.testing.assert_array_equal(grid.x_HII(), want["x_HII"])
    # FP32 deposits: at most 200 a cell here, each rounding by 2^-24 of the sum
    np.testing.assert_allclose(grid.rates()["kph"], ref.rates()["kph"], rtol=200 * 2.0 ** -24)
    grid.close()
    ref.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32_mixed"])
def test_rates_round_trip(precision):
    import torch
    dims = (5, 3, 7)
    n = int(np.prod(dims))
    grid = native.Grid(parity.ctx(), _medium(dims), precision)
    rng = np.random.default_rng(2)
    k = synth.round_f32(10.0 ** rng.uniform(-30, -8, n))
    gam = 10.0 ** rng.uniform(-44, -20, n)
    k[0] = gam[0] = 0.0
    native.rt_set_rates(grid.h, k, gam)
    for dtype, np_dtype in ((native.RT_DTYPE_F64, np.float64), (native.RT_DTYPE_F32, np.float32)):
        for where in ("host", "device"):
            r = native.rt_get_rates(grid.h, n, dtype, where)
            got = {q: np.asarray(v.cpu() if where == "device" else v) for q, v in r.items()}
            assert got["kph"].dtype == np_dtype
            np.testing.assert_array_equal(got["kph"], k.astype(np_dtype))
            # Gamma passes through FP32 eV/s on the mixed path and FP32 outputs (2^-24 each, and the
            # smallest FP32 number where it is subnormal)
            tol = 0.0 if precision == "fp64" and dtype == native.RT_DTYPE_F64 else 2.0 ** -22
            np.testing.assert_allclose(got["gamma"], gam, rtol=tol, atol=0.0 if tol == 0.0 else 1.5e-45)
    t = torch.tensor(k * 2, device="cuda")
    native.rt_set_rates(grid.h, t, torch.tensor(gam, device="cuda"))
    np.testing.assert_array_equal(grid.rates()["kph"], k * 2)
    grid.close()


@pytest.mark.parametrize("skip", [0, 1, 4])
@pytest.mark.parametrize("dims", [(3, 1, 1), (4, 1, 1), (5, 3, 7), (6, 8, 9)])
def test_fp32_rates_at_each_alignment(dims, skip):
    """Four cells a thread leave a remainder of 0 to 3, and an output may start
    off a 16-byte boundary.  k_ph is FP32 in the grid; Gamma leaves FP32 eV/s
    through an FP32 pair product instead of FP64: one FP32 rounding apart, or
    the smallest FP32 number where it is subnormal."""
    import torch
    n = int(np.prod(dims))
    grid = native.Grid(parity.ctx(), _medium(dims), "fp32_mixed")
    rng = np.random.default_rng(3)
    native.rt_set_rates(grid.h, synth.round_f32(10.0 ** rng.uniform(-30, -8, n)), 10.0 ** rng.uniform(-47, -20, n))
    want = grid.rates()
    out = torch.full((3, n + 8), -7.0, dtype=torch.float32, device="cuda")
    native.rt_get_rates_async(grid.h, *(out[q, skip:skip + n] for q in range(3)), dtype=native.RT_DTYPE_F32)
    native.rt_synchronize(grid.h)
    got = out.cpu().numpy()
    assert (got[:, :skip] == -7.0).all() and (got[:, skip + n:] == -7.0).all()
    np.testing.assert_array_equal(got[0, skip:skip + n], want["kph"].astype(np.float32))
    np.testing.assert_allclose(got[1, skip:skip + n], want["gamma"], rtol=2.0 ** -23, atol=1.5e-45)
    np.testing.assert_array_equal(got[2, skip:skip + n], want["x_HI"].astype(np.float32))
    grid.close()


@pytest.mark.parametrize("dims", [(1, 1, 1), (32, 8, 8), (33, 9, 9), (31, 7, 17), (3, 40, 2), (70, 1, 5)])
def test_timestep_on_partial_tiles(dims):
    g = _medium(dims, sources=1)
    grid, _, r = parity.run_gpu(g, "fp32_mixed")
    for kw in (dict(dt_max=1e16, tau_front=0.02), dict(dt_max=1e16, tau_front=0.0), dict(dt_max=1e16, tau_front=0.02)):
        want = timestep.rt_timestep(tuple(dims), g["box_len_cm"] / dims[0], g["n_H"], r["x_HI"],
                                    np.asarray(r["kph"], dtype=np.float64), **kw)
        assert native.rt_timestep(grid.h, **kw) == pytest.approx(want, rel=1e-5)
    grid.close()


@pytest.mark.parametrize("batched", [False, True])
def test_fp64_update_over_its_whole_range(batched):
    """Fractions, rates and densities inside and outside the range of the FP64
    update's FP32 guesses.  Each of the 10 substeps rounds by at most five
    units of 2^-53 on either side."""
    import oracle
    dims = (24, 20, 18)
    n = int(np.prod(dims))
    g = _medium(dims)
    rng = np.random.default_rng(6)
    small = 10.0 ** rng.uniform(-40, -0.31, n)
    x_small = rng.random(n) < 0.5
    g["x_HI"] = np.where(x_small, small, 1.0 - small)
    g["x_HII"] = np.where(x_small, 1.0 - small, small)
    g["n_H"] = 10.0 ** rng.uniform(-8, 12, n)
    k = np.where(rng.random(n) < 0.1, 0.0, 10.0 ** rng.uniform(-45, 8, n))
    grid = native.Grid(parity.ctx(), g, "fp64")
    native.rt_set_rates(grid.h, k, np.zeros(n))
    if batched:
        b = native.Batch(parity.ctx())
        b.add(grid)
        b.chem(synth.MYR_S, 10, synth.ALPHA_B)
    else:
        grid.chem(synth.MYR_S, 10, synth.ALPHA_B)
    x_o, z_o = oracle.chem(g["n_H"], g["x_HI"], g["x_HII"], k, synth.MYR_S, 10, synth.ALPHA_B)
    tol = 2 * 10 * 5 * 2.0 ** -53
    np.testing.assert_allclose(grid.rates()["x_HI"], x_o, rtol=tol, atol=0)
    np.testing.assert_allclose(grid.x_HII(), z_o, rtol=tol, atol=0)
    if batched:
        b.close()
    grid.close()


def _fp64_update(dims, n_H, x_HI, x_HII, k, dt_s, nsub, batched):
    g = _medium(dims)
    g.update(n_H=n_H, x_HI=x_HI, x_HII=x_HII)
    grid = native.Grid(parity.ctx(), g, "fp64")
    native.rt_set_rates(grid.h, k, np.zeros(k.size))
    if batched:
        b = native.Batch(parity.ctx())
        b.add(grid)
        b.chem(dt_s, nsub, synth.ALPHA_B)
        b.close()
    else:
        grid.chem(dt_s, nsub, synth.ALPHA_B)
    x, z = grid.rates()["x_HI"], grid.x_HII()
    grid.close()
    return x, z


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("nsub", [1, 2, 3])
def test_fp64_update_across_one_half(nsub, batched):
    """Few substeps over which the other fraction becomes the smaller one:
    neutral cells that are ionised, ionised cells that recombine.  Both keep
    five units of 2^-53 a substep on either side, relative."""
    import oracle
    dims = (16, 16, 16)
    n = int(np.prod(dims))
    rng = np.random.default_rng(12)
    h = synth.MYR_S / nsub
    ionise = np.arange(n) % 2 == 0
    small = np.where(rng.random(n) < 0.1, 0.0, 10.0 ** rng.uniform(-16, -0.31, n))
    x = np.where(ionise, 1.0 - small, small)
    z = np.where(ionise, small, 1.0 - small)
    a = 10.0 ** np.where(ionise, rng.uniform(-3, 2, n), rng.uniform(0, 7, n))  # h alpha_B n_H
    hk = np.where(ionise, 10.0 ** rng.uniform(0, 17, n), 0.0)
    n_H = a / (h * synth.ALPHA_B)
    got = _fp64_update(dims, n_H, x, z, hk / h, synth.MYR_S, nsub, batched)
    want = oracle.chem(n_H, x, z, hk / h, synth.MYR_S, nsub, synth.ALPHA_B)
    assert ((x > 0.5) != (want[0] > 0.5)).mean() > 0.5
    for q in range(2):
        np.testing.assert_allclose(got[q], want[q], rtol=2 * nsub * 5 * 2.0 ** -53, atol=0)


@pytest.mark.parametrize("nsub", [1, 2, 10])
def test_fp64_update_of_tiny_fractions(nsub):
    """Results down to 1e-60, where corrections held in FP32 would vanish:
    irradiated gas without recombination (no hydrogen, or next to none) and
    nearly neutral gas in the dark."""
    import oracle
    dims = (16, 16, 16)
    n = int(np.prod(dims))
    rng = np.random.default_rng(13)
    h = synth.MYR_S / nsub
    lit = np.arange(n) % 2 == 0
    small = 10.0 ** rng.uniform(-40, -10, n)
    x, z = np.where(lit, small, 1.0 - small), np.where(lit, 1.0 - small, small)
    hk = np.where(lit, 10.0 ** rng.uniform(-2, 17.5, n), 0.0)
    n_H = np.where(lit, np.where(rng.random(n) < 0.5, 0.0, 10.0 ** rng.uniform(-60, -20, n)),
                   10.0 ** rng.uniform(-3, 4, n))
    got = _fp64_update(dims, n_H, x, z, hk / h, synth.MYR_S, nsub, False)
    want = oracle.chem(n_H, x, z, hk / h, synth.MYR_S, nsub, synth.ALPHA_B)
    for q in range(2):
        np.testing.assert_allclose(got[q], want[q], rtol=2 * nsub * 5 * 2.0 ** -53, atol=0)


@pytest.mark.parametrize("nsub", [1, 3])
def test_fp64_update_of_unusual_states(nsub):
    """Both fractions as given, also where they do not add up to 1 (each
    rounded to FP32; apart by up to a tenth; x_HII not a number), and rates
    that are negative or not numbers: as the closed form has them."""
    import oracle
    dims = (16, 16, 16)
    n = int(np.prod(dims))
    rng = np.random.default_rng(14)
    h = synth.MYR_S / nsub
    kind = np.arange(n) % 4
    x = rng.uniform(0.01, 0.99, n)
    z = 1.0 - x
    x = np.where(kind == 0, synth.round_f32(x), x)
    z = np.where(kind == 0, synth.round_f32(z), np.where(kind == 1, z * rng.uniform(0.9, 1.1, n), z))
    a = 10.0 ** rng.uniform(-2, 2, n)
    hk = 10.0 ** rng.uniform(-3, 3, n)
    negative = kind == 2
    hk[negative] = rng.uniform(-0.3, 0.0, negative.sum())
    a[negative] = 10.0 ** rng.uniform(-4, -2, negative.sum())  # keeps the root real
    z[3], z[7], hk[11], hk[15] = np.nan, np.inf, np.nan, -np.inf
    n_H = a / (h * synth.ALPHA_B)
    got = _fp64_update(dims, n_H, x, z, hk / h, synth.MYR_S, nsub, False)
    want = oracle.chem(n_H, x, z, hk / h, synth.MYR_S, nsub, synth.ALPHA_B)
    for q in range(2):
        np.testing.assert_allclose(got[q], want[q], rtol=2 * nsub * 5 * 2.0 ** -53, atol=0)


@pytest.mark.parametrize("skip", [0, 1])
def test_rates_without_a_number_are_read_as_they_are(skip):
    """Infinities, values beyond FP32 and what is not a number, through both
    forms of the FP32 read."""
    import torch
    dims = (4, 3, 5)
    n = int(np.prod(dims))
    grid = native.Grid(parity.ctx(), _medium(dims), "fp32_mixed")
    gam = np.full(n, 1e-25)
    gam[1:8] = np.inf, -np.inf, np.nan, 1e60, -1e60, 3e26, -1e-25
    k = np.full(n, 1e-12)
    k[1:4] = np.inf, np.nan, 1e300
    native.rt_set_rates(grid.h, k, gam)
    want = grid.rates()
    assert np.isinf(want["gamma"][[1, 2, 4, 5]]).all() and np.isnan(want["gamma"][3])
    out = torch.zeros((2, n + 4), dtype=torch.float32, device="cuda")
    native.rt_get_rates_async(grid.h, *(out[q, skip:skip + n] for q in range(2)), dtype=native.RT_DTYPE_F32)
    native.rt_synchronize(grid.h)
    got = out.cpu().numpy()[:, skip:skip + n]
    np.testing.assert_array_equal(got[0], want["kph"].astype(np.float32))
    np.testing.assert_allclose(got[1], want["gamma"], rtol=2.0 ** -23)
    grid.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32_mixed"])
def test_device_arrays_off_an_element_boundary(precision):
    """Through the C ABI a device array may start at any byte: what kernels
    cannot read or write there is copied."""
    import torch
    dims = (5, 4, 3)
    n = int(np.prod(dims))
    grid = native.Grid(parity.ctx(), _medium(dims), precision)
    want = _medium(dims, seed=21)

    def put(a):
        t = torch.zeros(8 * n + 8, dtype=torch.uint8, device="cuda")
        t[4:4 + 8 * n] = torch.tensor(np.frombuffer(np.asarray(a, dtype=np.float64).tobytes(), dtype=np.uint8).copy())
        return t

    keep = [put(want["n_H"]), put(want["x_HI"])]
    native.check(native.lib().rt_set_state(grid.h, keep[0].data_ptr() + 4, keep[1].data_ptr() + 4, None,
                                           native.RT_MEM_DEVICE))
    bad = put(np.full(n, 2.0))
    with pytest.raises(native.RtError, match=r"x_HI\[0\]"):
        native.check(native.lib().rt_set_state(grid.h, None, bad.data_ptr() + 4, None, native.RT_MEM_DEVICE))
    rng = np.random.default_rng(3)
    k, gam = synth.round_f32(10.0 ** rng.uniform(-20, -8, n)), 10.0 ** rng.uniform(-30, -20, n)
    native.rt_set_rates(grid.h, k, gam)

    def read(field, dtype, off):  # one field into a buffer `off` bytes off
        size = 8 if dtype == native.RT_DTYPE_F64 else 4
        t = torch.full((size * n + 16,), 7, dtype=torch.uint8, device="cuda")
        p = [None, None, None]
        p[field] = t.data_ptr() + off
        native.check(native.lib().rt_get_rates_async(grid.h, *p, dtype, native.RT_MEM_DEVICE))
        native.rt_synchronize(grid.h)
        b = t.cpu().numpy()
        assert (b[:off] == 7).all() and (b[off + size * n:] == 7).all()
        return np.frombuffer(b[off:off + size * n].tobytes(), dtype=np.float64 if size == 8 else np.float32)

    np.testing.assert_array_equal(read(2, native.RT_DTYPE_F64, 4), want["x_HI"])
    if precision == "fp64":
        np.testing.assert_array_equal(read(0, native.RT_DTYPE_F64, 1), k)
        np.testing.assert_array_equal(read(1, native.RT_DTYPE_F64, 4), gam)
    else:
        np.testing.assert_array_equal(read(0, native.RT_DTYPE_F32, 2), k)
    grid.close()


@pytest.mark.parametrize("sdx,n_H,x,tau", [(7.0, 0.03, 0.2, None), (1e5, 1e25, 3e-40, None), (3.0, 1e37, 2e-42, None),
                                           (1e28, 1e-39, 0.3, None), (1e28, 1e-39, 0.3, 1e-20), (1e-28, 1e30, 0.5, None),
                                           (1e-20, 1e-25, 0.5, 1e-13), (1e29, 1e35, 1e-60, 1e3), (5.0, 1e-3, 1e-9, 0.0),
                                           (5.0, 1e-3, 0.0, 0.0), (2.0, 0.0, 0.5, 0.1)])
def test_front_cells_are_the_fp64_ones(sdx, n_H, x, tau):
    """One cell on either side of the threshold, from 1e-13 to 1e-3 of it (or at
    a threshold of its own), also where FP32 holds a factor to a few bits."""
    g = synth._grid((1, 1, 1), 1.0, 1.0, x, [[0.5, 0.5, 0.5]], [1e48], [13.6], [synth.SIGMA_HI])
    g["n_H"] = np.full(1, n_H)
    grid = native.Grid(parity.ctx(), g, "fp32_mixed")
    native.rt_set_rates(grid.h, np.full(1, 1e-10), np.zeros(1))
    depth = np.float64(sdx) * n_H * x
    steps = np.concatenate([s * 10.0 ** np.arange(-13, -2.9, 0.125) for s in (-1.0, 1.0)])
    for t in ([float(depth * (1.0 + d)) for d in steps] if tau is None else [tau]):
        got = native.rt_timestep(grid.h, sigma_front=sdx, tau_front=t, dt_max=1e20)
        assert (got < 1e19) == bool(depth > t), (t, got)  # 0.05 / rate in a front cell
    grid.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32_mixed"])
@pytest.mark.parametrize("dims", [(12, 16, 8), (13, 16, 8), (1, 1, 300), (1, 300, 1), (300, 1, 1), (2, 3, 200),
                                  (4, 4, 64), (3, 1, 90), (257, 2, 3)])
def test_timestep_of_thin_grids(precision, dims):
    """Grids that fill the tiles badly take two passes over a field: both forms
    against the oracle on either side of the rule."""
    g = _medium(dims, sources=1)
    grid, _, r = parity.run_gpu(g, precision)
    for kw in (dict(dt_max=1e16, tau_front=0.02), dict(dt_max=1e16, tau_front=0.0)):
        want = timestep.rt_timestep(tuple(dims), g["box_len_cm"] / dims[0], g["n_H"], r["x_HI"],
                                    np.asarray(r["kph"], dtype=np.float64), **kw)
        assert native.rt_timestep(grid.h, **kw) == pytest.approx(want, rel=1e-5)
    grid.close()


def test_timestep_takes_the_time_of_the_cells():
    """A column of cells is no slower than the same number in a cube by more
    than its neighbours' loads (five times allows for a slow call)."""
    import time
    best = []
    for dims in ((160, 160, 160), (1, 1, 4096000)):
        grid = native.Grid(parity.ctx(), synth._grid(dims, 1e21, 1e-3, 0.5, [[0, 0, 0]], [1e48], [13.6],
                                                     [synth.SIGMA_HI]), "fp32_mixed")
        n = int(np.prod(dims))
        native.rt_set_rates(grid.h, np.full(n, 1e-12), np.zeros(n))
        times = []
        for _ in range(8):
            t = time.perf_counter()
            native.rt_timestep(grid.h, dt_max=1e16)
            times.append(time.perf_counter() - t)
        best.append(min(times))
        grid.close()
    assert best[1] < 5 * best[0], best


@pytest.mark.parametrize("precision", ["fp64", "fp32_mixed"])
def test_host_reads_in_pieces(precision):
    """Fields longer than the read-back buffer (32 MB) by an odd remainder."""
    dims = (9000001, 1, 1)
    n = dims[0]
    grid = native.Grid(parity.ctx(), synth._grid(dims, 1e21, 1e-3, np.linspace(0.0, 1.0, n), [[0, 0, 0]], [1e48],
                                                 [13.6], [synth.SIGMA_HI]), precision)
    k = synth.round_f32(1e-12 * np.arange(1, n + 1))
    native.rt_set_rates(grid.h, k, k * 1e-13)
    for dtype, tol in ((native.RT_DTYPE_F64, 0.0 if precision == "fp64" else 2.0 ** -23), (native.RT_DTYPE_F32, 2.0 ** -22)):
        r = grid.rates(dtype)
        np.testing.assert_array_equal(r["kph"], k.astype(r["kph"].dtype))
        np.testing.assert_allclose(r["gamma"], k * 1e-13, rtol=tol)
        np.testing.assert_array_equal(r["x_HI"], np.linspace(0.0, 1.0, n).astype(r["x_HI"].dtype))
        np.testing.assert_array_equal(native.rt_get_ionised(grid.h, n, dtype),
                                      (1.0 - np.linspace(0.0, 1.0, n)).astype(r["x_HI"].dtype))
    grid.close()

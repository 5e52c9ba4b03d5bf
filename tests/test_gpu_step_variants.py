"""Launch rules and kernel variants of the step, at the sizes where they change:
every variant evaluates the per-node arithmetic of the two-pass form, so the
populations agree bit for bit."""
import numpy as np
import pytest
import torch

from paper_2101_04550_gb300 import elbm, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    elbm.load()


def field(lattice, n):
    if lattice == elbm.D3Q27:
        return inputs.isotropic_turbulence(n, seed=5, k0=3.0, u_rms=0.05)
    return inputs.double_shear_layer(n, U=0.08)


def populations(lattice, n, storage, kernel, steps, **kw):
    """Populations after the given launches of steps, from a seeded field."""
    rho, u = field(lattice, n)
    with elbm.Solver(lattice, n, storage=storage, kernel=kernel, T=0.42, nu=0.02,
                     stream=torch.cuda.current_stream(), **kw) as s:
        s.init(rho, u)
        for k in steps:
            s.step(k)
        return s.get_populations(dtype=np.float32)


# one plane per segment (32 x 16 x 3 is one tile column), a last segment
# shorter than the others (3 planes of 150), whole segments, the deepest ones
@pytest.mark.parametrize("n", [(32, 16, 3), (32, 16, 150), (64, 32, 33), (128, 80, 5), (512, 304, 70)])
@pytest.mark.parametrize("storage", [elbm.F32_SHIFT, elbm.F16_SHIFT])
def test_segment_depths_bitwise(n, storage):
    kw = dict(stretch=(1.0, 1.5, 2.0))
    want = populations(elbm.D3Q27, n, storage, 1, (1, 2), **kw)
    assert np.array_equal(populations(elbm.D3Q27, n, storage, 3, (1, 2), **kw), want)


@pytest.mark.parametrize("n", [(32, 8, 3), (64, 24, 41)])
def test_segment_depths_of_eight_row_tiles_bitwise(n):
    want = populations(elbm.D3Q27, n, elbm.F32, 1, (3,))
    assert np.array_equal(populations(elbm.D3Q27, n, elbm.F32, 3, (3,)), want)


# the gradient pass takes four nodes at once where rows allow it, the mode sums 32 x 64
# nodes of a plane: grids inside that, one node past it, and ragged along every axis;
# one array at both streaming parities
@pytest.mark.parametrize("lattice,n", [(elbm.D3Q27, (5, 3, 70)), (elbm.D3Q27, (33, 9, 3)), (elbm.D3Q27, (97, 65, 4)),
                                       (elbm.D2Q9, (33, 5)), (elbm.D2Q9, (300, 130))])
@pytest.mark.parametrize("steps,walls", [(0, False), (1, False), (1, True), (2, True)])
def test_diagnostics_against_the_read_out_fields(lattice, n, steps, walls):
    """Reductions and mode amplitude against FP64 sums over the fields that
    elbm_moments returns.  A term of a sum carries at most 8 FP32 roundings, so
    a sum is within 8 * 2^-24 of the sum of its terms' absolute values."""
    lam, D = (1.0, 1.5, 2.0), 3 if lattice == elbm.D3Q27 else 2
    rho, u = field(lattice, n)
    with elbm.Solver(lattice, n, stretch=lam, T=0.42, nu=0.02, storage=elbm.F32_SHIFT, kernel=1, walls_y=walls,
                     force=(1e-4, 0.0, 0.0)[:D]) as s:
        s.init(rho, u)
        s.step(steps)
        red = s.reduce()
        k = [2 * np.pi / (n[a] * lam[a]) for a in range(D)]
        amp = s.mode_amplitude(k, (0.3, -0.8, 0.5)[:D])
        f = s.get_populations()
        r32, u32 = s.moments(dtype=np.float32)
    r, v = r32.astype(np.float64), u32.astype(np.float64)

    def diff(w, a):
        ax = w.ndim - 1 - a
        up, dn = np.roll(w, -1, ax), np.roll(w, 1, ax)
        if walls and a == 1:
            up = np.concatenate([np.delete(w, 0, ax), -w.take([-1], ax)], ax)
            dn = np.concatenate([-w.take([0], ax), np.delete(w, -1, ax)], ax)
        return (up - dn) / (2 * lam[a]), (np.abs(up) + np.abs(dn)) / (2 * lam[a])

    def close(got, terms, bound=None):
        assert abs(got - terms.sum()) <= 8 * 2.0 ** -24 * (np.abs(terms) if bound is None else bound).sum()

    u2 = (v ** 2).sum(0)
    close(red["mass"], r)
    for a, name in enumerate(("mom_x", "mom_y", "mom_z")[:D]):
        close(red[name], r * v[a])
    close(red["rho_u2"], r * u2)
    close(red["u2"], u2)
    close(red["ux2"], v[0] ** 2)
    pairs = [(1, 0, 0, 1)] + ([(2, 1, 1, 2), (0, 2, 2, 0)] if D == 3 else [])
    curl, size = 0.0, 0.0
    for a, da, b, db in pairs:
        (x, ax_), (y, ay_) = diff(v[a], da), diff(v[b], db)
        curl, size = curl + (x - y) ** 2, size + (ax_ + ay_) ** 2
    close(red["curl2"], curl, size)
    dx, size = diff(v[0], 0)
    close(red["dxux2"], dx ** 2, size ** 2)
    assert red["umax"] == pytest.approx(np.sqrt(u2.max()), rel=1e-6)
    assert red["fmin"] == pytest.approx(f.min(), rel=1e-5)
    assert red["nonfinite"] == 0
    if walls:
        ux = np.moveaxis(v[0], v[0].ndim - 2, 0)
        close(red["wall_dudn"], (9 * ux[[0, -1]] - ux[[1, -2]]) / (3 * lam[1]),
              (9 * np.abs(ux[[0, -1]]) + np.abs(ux[[1, -2]])) / (3 * lam[1]))
    phase = sum(np.arange(n[a]).reshape([-1 if d == D - 1 - a else 1 for d in range(D)]) * lam[a] * k[a]
                for a in range(D))
    us = sum(v[a] * w for a, w in zip(range(D), (0.3, -0.8, 0.5)))
    want = 2 * abs((us * np.exp(-1j * phase)).sum()) / r.size
    assert abs(amp - want) <= 8 * 2.0 ** -24 * 2 * np.abs(us).mean() + 1e-15


# the 64-wide tiles (8 rows) of the TMEM single pass beside the 32-wide ones (16
# rows), with one tile buffer and with two: one tile column that wraps onto itself,
# a single row of tiles, sizes past 2^18 nodes; FX the force along x alone
@pytest.mark.parametrize("n", [(64, 16, 3), (64, 48, 9), (192, 16, 5), (96, 32, 7), (160, 64, 27), (128, 128, 19)])
@pytest.mark.parametrize("storage", [elbm.F32, elbm.F32_SHIFT, elbm.F16_SHIFT, elbm.BF16_SHIFT])
@pytest.mark.parametrize("opts", [{}, {"walls_y": True, "force": (1e-5, 0.0, 0.0)},
                                  {"walls_y": True, "force": (1e-5, 2e-6, -3e-6)}])
def test_tile_shapes_bitwise(n, storage, opts):
    kw = dict(stretch=(1.5, 1.0, 2.0), **opts)
    want = populations(elbm.D3Q27, n, storage, 1, (1, 2), **kw)
    assert np.array_equal(populations(elbm.D3Q27, n, storage, 3, (1, 2), **kw), want)


# the cp.async-fed single pass (any grid): smaller than a tile, one node more or
# less than one, 64-wide and 32-wide tiles, rows on 16 bytes and on 4 and 2
@pytest.mark.parametrize("n", [(3, 3, 3), (31, 15, 4), (33, 17, 5), (65, 9, 3), (128, 10, 6), (36, 24, 41), (100, 50, 9),
                               (95, 33, 6), (180, 30, 12)])
@pytest.mark.parametrize("storage", [elbm.F32, elbm.F32_SHIFT, elbm.F16_SHIFT, elbm.BF16_SHIFT])
def test_single_pass_on_any_grid_bitwise(n, storage):
    kw = dict(stretch=(1.5, 1.0, 2.0))
    want = populations(elbm.D3Q27, n, storage, 1, (1, 2, 4), **kw)
    assert np.array_equal(populations(elbm.D3Q27, n, storage, 3, (1, 2, 4), **kw), want)


def test_single_pass_repeats_its_bits():
    """Many short runs of the single pass, step launches overlapping, give the
    same bits every time (a buffer handed back early shows as a rare difference)."""
    n = (96, 32, 40)
    rho, u = field(elbm.D3Q27, n)
    rho, u = torch.tensor(rho, device="cuda"), torch.tensor(u, device="cuda")
    for storage in (elbm.F32_SHIFT, elbm.F16_SHIFT):
        got = []
        for kernel, runs in ((1, 1), (3, 400)):
            with elbm.Solver(elbm.D3Q27, n, storage=storage, kernel=kernel, T=0.42, nu=0.02,
                             stream=torch.cuda.current_stream()) as s:
                out = torch.empty((27,) + n[::-1], device="cuda")
                for _ in range(runs):
                    s.init(rho, u)
                    s.step(27)
                    s.get_populations(out)
                    if kernel == 3:
                        assert torch.equal(out, got[0])
                got.append(out.clone())


# small D2Q9 grids, several steps a launch in one cluster: one to eight bands of
# rows, a short last band, several nodes a thread, 16-bit rows; single steps between
@pytest.mark.parametrize("n", [(3, 3), (64, 64), (33, 5), (100, 37), (17, 129), (500, 18), (1536, 8), (1537, 8)])
@pytest.mark.parametrize("storage", [elbm.F32, elbm.F32_SHIFT, elbm.F16_SHIFT, elbm.BF16_SHIFT])
@pytest.mark.parametrize("equilibrium", [0, 1])
def test_small_d2q9_bitwise(n, storage, equilibrium):
    kw = dict(stretch=(1.5, 1.0), equilibrium=equilibrium)
    want = populations(elbm.D2Q9, n, storage, 1, (2, 1, 33), **kw)
    assert np.array_equal(populations(elbm.D2Q9, n, storage, 3, (2, 1, 33), **kw), want)


# the reductions' compensated sums over many nodes a thread: 64-bit sums of the same
# FP32 terms.  A thread's sum is within kFold n 2^-49 of its terms' magnitudes (kFold = 8
# terms between folds, n terms), the FP64 sums add less than 2^-40.
@pytest.mark.parametrize("tail", [2.9e-9, 3.1e-9, 3.4e-9])
def test_sum_of_a_large_term_and_many_small_ones(tail):
    """A jet in the rows that are every thread's first node, a nearly quiescent
    field behind it: a thread adds hundreds of terms below half a unit in the
    last place of its sum."""
    N = 8192
    u = torch.zeros((2, N, N), device="cuda")
    u[0] = tail
    u[0, :14] = 0.1   # 114688 nodes; the reduction has some 117000 threads
    with elbm.Solver(elbm.D2Q9, (N, N), storage=elbm.F32_SHIFT, kernel=1, T=0.42, nu=0.02,
                     stream=torch.cuda.current_stream()) as s:
        s.init(torch.ones((N, N), device="cuda"), u)
        red = s.reduce()
        rho = torch.empty((N, N), device="cuda")
        s.moments(rho, u)
        terms = rho * u[0]   # in FP32, as the kernel forms them
    want, size = float(terms.double().sum()), float(terms.double().abs().sum())
    n = -(-N * N // 114688)
    assert abs(red["mom_x"] - want) <= (8 * n * 2.0 ** -49 + 2.0 ** -40) * size


# read-outs of one array at odd parity (bounced slots with walls, none without) against
# the own-location layout of the single pass: the same state, so the same bits
@pytest.mark.parametrize("lattice,n,walls", [(elbm.D3Q27, (64, 32, 9), False), (elbm.D3Q27, (64, 32, 9), True),
                                             (elbm.D2Q9, (65, 33), False)])
@pytest.mark.parametrize("storage", [elbm.F32, elbm.F32_SHIFT, elbm.F16_SHIFT, elbm.BF16_SHIFT])
def test_read_outs_at_odd_parity(lattice, n, walls, storage):
    rho, u = field(lattice, n)
    got = []
    for kernel in (1, 3):
        with elbm.Solver(lattice, n, storage=storage, kernel=kernel, T=0.42, nu=0.02, walls_y=walls) as s:
            s.init(rho, u)
            s.step(3)
            r, v = s.moments(dtype=np.float32)
            got.append((r, v, s.get_populations(), s.reduce(), s.mode_amplitude((0.3, 0.2, 0.1), (0.4, -0.5, 0.6))))
    for a, b in zip(*got):
        assert a == b if isinstance(a, (dict, float)) else np.array_equal(a, b)


# the reductions of grids of several nodes a thread (rows in 16-byte pieces and not), and
# the mode sums node by node on planes smaller than a block's columns and rows
@pytest.mark.parametrize("n", [(96, 80, 64), (97, 81, 64), (3, 4, 40000), (12, 9, 5000)])
@pytest.mark.parametrize("steps,walls", [(0, False), (1, True)])
def test_diagnostics_of_several_nodes_a_thread(n, steps, walls):
    test_diagnostics_against_the_read_out_fields(elbm.D3Q27, n, steps, walls)


def test_diagnostics_count_non_finite_nodes():
    """A NaN and an infinite population: counted, left out of the extrema, and
    reported; the sums over them are not finite."""
    n = (96, 80, 64)
    rho, u = field(elbm.D3Q27, n)
    with elbm.Solver(elbm.D3Q27, n, storage=elbm.F32, kernel=1, T=0.42, nu=0.02) as s:
        s.init(rho, u)
        f = s.get_populations()
        f[3, 0, 0, 5] = np.nan
        f[13, 63, 79, 95] = np.inf
        s.set_populations(f)
        red = s.reduce(raise_nonfinite=False)
        with pytest.raises(elbm.ElbmError) as err:
            s.reduce()
        r, v = s.moments(dtype=np.float32)
    bad = ~np.isfinite(f).all(0)
    assert err.value.code == -5 and bad.sum() == 2
    assert red["nonfinite"] == 2 and not np.isfinite(red["mass"])
    assert red["umax"] == pytest.approx(np.sqrt((v[:, ~bad].astype(np.float64) ** 2).sum(0).max()), rel=1e-6)
    assert red["fmin"] == pytest.approx(f[:, ~bad].min(), rel=1e-5)


# which calls the cluster takes, by their launches: one to three nodes a thread, the
# fewest steps of each and one less, three blocks and eight, more of the march's blocks
# than SMs, more steps than one launch takes, a grid too large
@pytest.mark.parametrize("n,steps,launches", [((64, 64), 1, 1), ((64, 64), 2, 1), ((512, 3), 2, 2), ((512, 3), 3, 1),
                                              ((128, 64), 4, 4), ((128, 64), 5, 1), ((192, 64), 7, 7),
                                              ((192, 64), 8, 1), ((1536, 3), 15, 15), ((1536, 3), 16, 1),
                                              ((12, 1000), 2, 1), ((33, 5), 4099, 2), ((1537, 8), 33, 33)])
def test_small_d2q9_calls(n, steps, launches):
    rho, u = field(elbm.D2Q9, n)
    with elbm.Solver(elbm.D2Q9, n, kernel=3, T=0.42, nu=0.02, stream=torch.cuda.current_stream()) as s:
        s.init(rho, u)
        before = s.launches
        s.step(steps)
        assert s.launches - before == launches
        got = s.get_populations()
    assert np.array_equal(got, populations(elbm.D2Q9, n, elbm.F32, 1, (steps,)).astype(np.float64))

"""Terms of the field against extended precision where one of them, or one
component, is far smaller or larger than the rest: each has to be as accurate
as its own arithmetic, not only as the whole field's largest term."""
import numpy as np
import pytest
import torch

from oracle import micromag as om
from gpu_cases import dev, make_pair

pytestmark = pytest.mark.gpu
LD = np.longdouble
AXES = ((3, "dx"), (2, "dy"), (1, "dz"))


def smooth(shape, seed):
    """Three smooth fields of order one."""
    z, y, x = np.meshgrid(*(np.linspace(0.0, 1.0, n) for n in shape), indexing="ij")
    r = np.random.default_rng(seed).uniform(0.5, 2.0, (3, 4))
    return np.stack([np.cos(a * x + b * y + c * z + d) for a, b, c, d in r])


def exchange(p, m):
    """The exchange field in extended precision, and the sum of its terms' magnitudes."""
    M = m.astype(LD)
    H, mag = np.zeros_like(M), np.zeros_like(M)
    for ax, d in AXES:
        if m.shape[ax] < 2:
            continue
        c = LD(2) * LD(p.A) / (LD(om.MU0) * LD(p.Ms) * LD(getattr(p, d)) ** 2)
        diff = c * np.diff(M, axis=ax)
        for sign, pad in ((1, (0, 1)), (-1, (1, 0))):
            t = np.pad(sign * diff, [pad if a == ax else (0, 0) for a in range(4)])
            H += t
            mag += abs(t)
    return H, mag


def field(mmlib, prob, m, Hext, dtype=torch.float64):
    H = torch.empty(m.shape, dtype=dtype, device="cuda")
    mmlib.mm_heff(prob, dev(m, dtype), Hext, H)
    return H.cpu().numpy()


@pytest.mark.parametrize("grid", [(1, 9, 1), (24, 7, 1), (9, 1, 2), (33, 18, 3), (9, 6, 7)])
def test_exchange_of_a_small_component_beside_a_large_one(mmlib, grid):
    """Differences of doubles this close are exact, so a cell's sum is off by the roundings of at most six terms: three
    roundings each at the terms' size, 18 x 2^-53 < 2^-48 of the sum of their magnitudes.  The coefficient's own rounding
    adds three, the demagnetisation (2^-50 Ms) nothing: the exchange field is 10^4 Ms and more here."""
    nx, ny, nz = grid
    prob, p = make_pair(mmlib, nx, ny, nz, (1e-9, 1.1e-9, 0.9e-9), Ms=1e3, A=1e-11, K=0.0)
    for big in range(3):
        m = 1e-6 * smooth(p.shape, 7 + big)
        m[big] = 1.0
        H = field(mmlib, prob, m, (0, 0, 0))
        ref, mag = exchange(p, m)
        ref = ref + om.Demag(p).field(m)
        assert np.all(abs(H - ref) <= 2.0 ** -48 * mag + 2.0 ** -49 * p.Ms)


@pytest.mark.parametrize("prec,dtype,h", [("MM_FP64", torch.float64, 2.0 ** 42), ("MM_FP32", torch.float32, 2.0 ** 34)])
@pytest.mark.parametrize("grid", [(24, 7, 1), (9, 6, 3), (8, 9, 7)])
def test_large_external_field_is_rounded_once(mmlib, grid, prec, dtype, h):
    """The other terms (below 2^22 A/m) are summed first: a component is off by half a unit in the last place of the
    external field and the terms' own error, at most 2^-42 (FP64) and 2^-16 (FP32) of 2^22."""
    nx, ny, nz = grid
    prob, p = make_pair(mmlib, nx, ny, nz, (4e-9, 3e-9, 5e-9), A=1.3e-11, K=2e4, u=(0.6, 0.0, 0.8),
                        precision=getattr(mmlib, prec))
    m = smooth(p.shape, 3)
    m = (m / np.sqrt((m * m).sum(0))).astype(np.float32).astype(np.float64)
    ref = om.heff(p, m, np.zeros(3), om.Demag(p))
    assert np.max(abs(ref)) < 2.0 ** 22
    Hext = np.array([1.25 * h, -1.5 * h, 1.75 * h])      # exact in either type; sums stay in the same binade
    H = field(mmlib, prob, m, Hext, dtype).astype(LD)
    ulp = h * 2.0 ** (-52 if prec == "MM_FP64" else -23)
    own = 2.0 ** 22 * (2.0 ** -42 if prec == "MM_FP64" else 2.0 ** -16)
    assert np.max(abs(H - (ref.astype(LD) + Hext.reshape(3, 1, 1, 1)))) <= 0.5 * ulp + own


@pytest.mark.parametrize("prec,u,floor", [("MM_FP64", 2.0 ** -53, 2.0 ** -50), ("MM_F32X2", 2.0 ** -47, 2.0 ** -44),
                                          ("MM_FP32", 2.0 ** -24, 2.0 ** -20)])
@pytest.mark.parametrize("Ms,K,tilt", [(1.28e6, 4.3e6, 0.1), (3e5, 6e6, 1e-3), (8e5, 500.0, 0.1)])
def test_energy_of_a_minimisation_with_a_large_uniform_anisotropy(mmlib, Ms, K, tilt, prec, u, floor):
    """The cells' anisotropy terms cancel against 2 K/(mu0 Ms) before they are summed, so what is left of K V N in the
    sum is each cell's own rounding: about 4 u K V, of either sign, 16 u K V N / sqrt(N) at four standard deviations.
    `floor` covers the other terms."""
    nx, ny, nz = 256, 128, 2
    N = nx * ny * nz
    cell = (4e-9, 4e-9, 5e-9)
    single = prec == "MM_FP32"
    Hext = np.array([5e4, 0.0, 2e4])
    m = tilt * np.random.default_rng(5).standard_normal((3, nz, ny, nx))
    m[0] += 1.0
    m /= np.sqrt((m * m).sum(0))
    m = m.astype(np.float32).astype(np.float64) if single else m
    prob, p = make_pair(mmlib, nx, ny, nz, cell, Ms=Ms, A=1e-11, K=K, precision=getattr(mmlib, prec))
    _, r = mmlib.mm_minimize(prob, dev(m, torch.float32 if single else torch.float64), Hext, mmlib.make_opts(max_iter=0))
    double, _ = make_pair(mmlib, nx, ny, nz, cell, Ms=Ms, A=1e-11, K=K)
    M, V, c = m.astype(LD), LD(cell[0]) * LD(cell[1]) * LD(cell[2]), LD(om.MU0) * LD(Ms)
    ref = LD(mmlib.mm_energy(double, dev(m), Hext)[0]) - c * V / 2 * (M * exchange(p, m)[0]).sum()
    ref += LD(K) * V * (1 - M[0] ** 2).sum() - c * V * (M * Hext.astype(LD).reshape(3, 1, 1, 1)).sum()
    assert abs(r.energy - ref) <= 16 * u * float(K * V) * N ** 0.5 + floor * float(abs(ref))


def coupled(shape, a, b):
    """Whether the tensor mixes components a and b: the cells of an axis lie on both sides of one another."""
    n = shape[::-1]
    return a == b or (n[a] > 1 and n[b] > 1)


@pytest.mark.parametrize("prec,bar", [("MM_FP64", 2e-15), ("MM_F32X2", 1e-13)])
@pytest.mark.parametrize("grid", [(24, 20, 1), (1, 36, 1), (300, 1, 1), (24, 1, 3), (1, 20, 2), (257, 9, 1), (12, 1, 9),
                                  (1, 1, 24), (1, 9, 70)])
def test_components_of_different_size(mmlib, grid, prec, bar):
    """A magnetisation tilted by little from an axis: the field of the components that the tensor does not mix with the
    large one is as accurate as that of components of their own size (the bars of random states, relative to Ms times
    the mixed components: the field itself can be a small difference).  The tilts stay far above the oracle's tensor
    entries of pairs that do not mix, 1e-33 in place of 0."""
    nx, ny, nz = grid
    if prec == "MM_F32X2" and nz > 4:
        pytest.skip("double-word problems are films")
    prob, p = make_pair(mmlib, nx, ny, nz, (4e-9, 3e-9, 5e-9), A=0.0, K=0.0, precision=getattr(mmlib, prec))
    d = om.Demag(p)
    for big in range(3):
        for tilt in (1e-3, 1e-8, 1e-12):
            m = tilt * smooth(p.shape, 11 + big)
            m[big] = 1.0
            H, ref = field(mmlib, prob, m, (0, 0, 0)), d.field(m)
            for c in range(3):
                mixed = np.sqrt(sum(np.sum(m[a] ** 2) for a in range(3) if coupled(p.shape, a, c)))
                assert np.linalg.norm(H[c] - ref[c]) <= bar * p.Ms * mixed, (big, tilt, c)


def test_grouped_batch_with_grids_of_one_row_or_column_equals_single_sweeps(mmlib):
    sizes = [(24, 1, 3), (1, 20, 2), (16, 9, 2), (40, 1, 1), (1, 150, 4), (12, 10, 4)]
    probs = [make_pair(mmlib, *n, (4e-9, 3e-9, 5e-9))[0] for n in sizes]
    F = np.array([[2e4, 1e3, 0.0], [-1e4, 1e3, 0.0]])
    opts = mmlib.make_opts(max_iter=6)
    batch = mmlib.mm_batch_create(probs, mmlib.MM_BATCH_GROUPED)
    starts = [smooth((nz, ny, nx), 5 + nx) for nx, ny, nz in sizes]
    starts = [dev(m / np.sqrt((m * m).sum(0))) for m in starts]
    ms = [m.clone() for m in starts]
    _, mavg, _ = mmlib.mm_batch_sweep(batch, ms, F, opts=opts)
    for i, p in enumerate(probs):
        _, mavg1, _ = mmlib.mm_hysteresis_sweep(p, starts[i], F, opts=opts)
        assert torch.equal(ms[i], starts[i]) and np.array_equal(mavg[i], mavg1), sizes[i]
    batch.close()


@pytest.mark.parametrize("prec,bar", [("MM_FP64", 2e-15), ("MM_F32X2", 1e-13)])
def test_field_does_not_depend_on_the_tile_chosen_by_timing(mmlib, prec, bar):
    """Rows of very different magnitude (as the Hessian product and the adjoint evaluate): problems of one grid, whose
    tiles are timed anew at each setup, and a repeated evaluation give the same bits, and the rows' scales the accuracy
    of one scale."""
    grid = (130, 128, 4)   # above the size from which tiles are timed
    m = smooth((4, 128, 130), 9) * 2.0 ** (-3.0 * (np.arange(128) % 13)).reshape(1, 1, 128, 1)
    fields, tiles = [], set()
    for _ in range(6):
        prob, p = make_pair(mmlib, *grid, (4e-9, 3e-9, 5e-9), A=0.0, K=0.0, precision=getattr(mmlib, prec))
        tiles.add(mmlib.mm_problem_info(prob)["x_fwd_tile_rows"])
        fields += [field(mmlib, prob, m, (0, 0, 0)) for _ in range(2)]
        prob.close()
    assert all(np.array_equal(f, fields[0]) for f in fields), tiles
    ref = om.Demag(p).field(m)
    assert np.linalg.norm(fields[0] - ref) <= bar * p.Ms * np.linalg.norm(m)


@pytest.mark.parametrize("prec,bar", [("MM_FP64", 2e-15), ("MM_F32X2", 1e-13)])
@pytest.mark.parametrize("cell", [(4e-9, 4e-9, 4e-13), (4e-13, 3e-9, 4e-9), (4e-9, 2e-10, 5e-9)])
@pytest.mark.parametrize("grid", [(24, 20, 1), (40, 1, 1), (18, 12, 2), (12, 10, 4), (1, 20, 3), (8, 9, 7), (12, 1, 9)])
def test_flat_cells(mmlib, grid, cell, prec, bar):
    """Cells whose tensor has elements far below its largest: every component is accurate to the products that form it.
    The bars are those of random states, relative to the sum over the components of the largest modulus of the element's
    transform times the component."""
    nx, ny, nz = grid
    if prec == "MM_F32X2" and nz > 4:
        pytest.skip("double-word problems are films")
    prob, p = make_pair(mmlib, nx, ny, nz, cell, A=0.0, K=0.0, precision=getattr(mmlib, prec))
    d = om.Demag(p)
    top = [[p.Ms * np.max(abs(N)) for N in row] for row in om._sym(d.Nhat)]
    for big in range(3):
        for tilt in (0.3, 1e-8):
            m = tilt * smooth(p.shape, 11 + big)
            m[big] = 1.0
            H, ref = field(mmlib, prob, m, (0, 0, 0)), d.field(m)
            for c in range(3):
                terms = sum(top[c][b] * np.linalg.norm(m[b]) for b in range(3) if coupled(p.shape, b, c))
                assert np.linalg.norm(H[c] - ref[c]) <= bar * terms, (big, tilt, c)


@pytest.mark.parametrize("prec", ["MM_FP64", "MM_FP32", "MM_F32X2"])
def test_nothing_of_the_timed_state_stays_behind(mmlib, prec):
    """Launch shapes are timed at setup on a field of the tuner's own: a new problem holds zeros."""
    dt = torch.float32 if prec == "MM_FP32" else torch.float64
    prob, p = make_pair(mmlib, 130, 128, 4, (4e-9, 3e-9, 5e-9), precision=getattr(mmlib, prec))
    bufs = [torch.ones((3,) + p.shape, dtype=dt, device="cuda") for _ in range(4)]
    st = mmlib.mm_min_inspect(prob, *bufs)
    assert all(not b.any() for b in bufs)
    info = mmlib.mm_problem_info(prob)
    assert info["x_tile_rows"] in (1, 2, 4, 8, 16) and info["x_fwd_tile_rows"] in (1, 2, 4, 8, 16)
    assert 12 % info["yz_batch_rows"] == 0 and st is not None

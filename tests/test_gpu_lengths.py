"""Padded lengths with odd parts (5/8, 3/4 and 25/32 of a power of two): the
field of every such length along each axis, in each precision and layout,
against the oracle's FFT on its own padding (2n per axis).

Bars as for the powers of two: FP64 2e-15 and FP32 3e-6 rel-L2 of the
demagnetisation field of a random state, double-word 1e-13 (about 2^-47 per
element times the root of the number of passes)."""
import numpy as np
import pytest
import torch

from oracle import micromag as om
from paper_1405_2728_gb300 import inputs
from gpu_cases import dev, make_pair, rel_l2

pytestmark = pytest.mark.gpu
CELL = (3.90625e-9, 3.90625e-9, 5e-9)
# cells -> padded length: x, and y of films; y and z of bulk grids
FILM = {128: 256, 129: 320, 160: 320, 161: 384, 192: 384, 193: 512, 257: 640, 320: 640, 384: 768, 385: 1024}
BULK = {32: 64, 33: 80, 40: 80, 48: 96, 49: 128, 80: 160, 96: 192, 100: 200, 101: 256, 160: 320, 192: 384, 200: 400, 320: 640,
        384: 768, 400: 800}


def demag_error(mmlib, grid, prec):
    nx, ny, nz = grid
    prob, oprob = make_pair(mmlib, nx, ny, nz, CELL, A=0.0, K=0.0, precision=getattr(mmlib, prec))
    dt = torch.float32 if prec == "MM_FP32" else torch.float64
    m = inputs.random_unit_m(oprob.shape, 17 + nx + ny + nz)
    if prec == "MM_FP32":
        m = m.astype(np.float32).astype(np.float64)
    H = torch.empty(m.shape, dtype=dt, device="cuda")
    mmlib.mm_heff(prob, dev(m, dt), (0, 0, 0), H)
    info = mmlib.mm_problem_info(prob)
    prob.close()
    return rel_l2(H.cpu().numpy(), om.Demag(oprob).field(m)), info


BAR = {"MM_FP64": 2e-15, "MM_FP32": 3e-6, "MM_F32X2": 1e-13}


@pytest.mark.parametrize("prec", ["MM_FP64", "MM_FP32", "MM_F32X2"])
@pytest.mark.parametrize("n", sorted(FILM))
def test_film_axes(mmlib, n, prec):
    err, info = demag_error(mmlib, (n, 5, 1 + n % 4), prec)
    assert info["px"] == FILM[n] and info["bulk_layout"] == 0
    assert err <= BAR[prec]
    err, info = demag_error(mmlib, (6, n, 1 + n % 3), prec)
    assert info["py"] == FILM[n] and info["bulk_layout"] == 0
    assert err <= BAR[prec]


@pytest.mark.parametrize("prec", ["MM_FP64", "MM_FP32"])
@pytest.mark.parametrize("n", sorted(BULK))
def test_bulk_axes(mmlib, n, prec):
    err, info = demag_error(mmlib, (5, n, 6), prec)
    assert info["py"] == BULK[n] and info["bulk_layout"] == 1
    assert err <= BAR[prec]
    err, info = demag_error(mmlib, (4, 7, n), prec)
    assert info["pz"] == BULK[n] and info["bulk_layout"] == 1
    assert err <= BAR[prec]


def test_layout_and_support_do_not_depend_on_the_padding(mmlib):
    """A film whose power-of-two plane does not fit one CTA stays in the bulk layout, and is still refused in double-word
    precision."""
    grid = mmlib.make_grid(40, 300, 4, *CELL)   # pads to 640, whose plane would fit; 1024 does not
    p = mmlib.mm_setup_geometry(grid, mmlib.make_material(8e5, 1.3e-11, 500.0), mmlib.MM_FP64)
    info = mmlib.mm_problem_info(p)
    assert info["bulk_layout"] == 1 and info["py"] == 640
    with pytest.raises(mmlib.MMError) as e:
        mmlib.mm_setup_geometry(grid, mmlib.make_material(8e5, 1.3e-11, 500.0), mmlib.MM_F32X2)
    assert e.value.status == mmlib.MM_ERR_UNSUPPORTED


@pytest.mark.parametrize("prec", ["MM_FP64", "MM_FP32"])
def test_grouped_batch_of_such_films_equals_single_sweeps(mmlib, prec):
    # every odd y length of films (320, 384, 640, 768), both size groups: the grouped kernels give the
    # films' own results bit for bit
    sizes = [(24, 150, 1), (20, 190, 2), (16, 300, 3), (12, 350, 1), (160, 130, 4)]
    dt = torch.float32 if prec == "MM_FP32" else torch.float64
    probs = [mmlib.mm_setup_geometry(mmlib.make_grid(*n, *CELL), mmlib.make_material(8e5, 1.3e-11, 500.0),
                                     getattr(mmlib, prec)) for n in sizes]
    assert [mmlib.mm_problem_info(p)["py"] for p in probs] == [320, 384, 640, 768, 320]
    F = np.array([[2e4, 1e3, 0.0], [-1e4, 1e3, 0.0]])
    opts = mmlib.make_opts(max_iter=6)
    batch = mmlib.mm_batch_create(probs, mmlib.MM_BATCH_GROUPED)
    starts = [dev(inputs.random_unit_m((nz, ny, nx), 5 + nx), dt) for nx, ny, nz in sizes]
    ms = [m.clone() for m in starts]
    _, mavg, _ = mmlib.mm_batch_sweep(batch, ms, F, opts=opts)
    for i, p in enumerate(probs):
        _, mavg1, _ = mmlib.mm_hysteresis_sweep(p, starts[i], F, opts=opts)
        assert torch.equal(ms[i], starts[i]) and np.array_equal(mavg[i], mavg1), sizes[i]
    batch.close()

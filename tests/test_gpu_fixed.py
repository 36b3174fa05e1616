"""The block fixed-point convolution of MM_FP64 (csrc/fixed.cuh): its scaling
over field magnitudes, its edges of sizes and layer counts, and non-finite
inputs.

Bars.  Against the oracle's double FFT: a double FFT's own error is about
2^-52 times a small multiple of sqrt(log2 N) in the 2-norm and the fixed-point
one keeps up to 58 bits per block, so 2e-15 rel-L2 leaves a factor of 4 for
both together.  A power of two in m enters only the blocks' exponents, so it
comes out exactly."""
import numpy as np
import pytest
import torch

from oracle import micromag as om
from paper_1405_2728_gb300 import inputs
from gpu_cases import dev, make_pair, rel_l2

pytestmark = pytest.mark.gpu
CELL = (3.90625e-9, 3.90625e-9, 5e-9)


def demag(mmlib, prob, m):
    H = torch.empty(m.shape, dtype=torch.float64, device="cuda")
    mmlib.mm_heff(prob, dev(m), (0, 0, 0), H)
    return H.cpu().numpy()


# row lengths below 8, of every radix mix, compiled and general; 1 to 4 layers; bulk grids with ragged blocks
@pytest.mark.parametrize("grid", [(1, 1, 1), (2, 2, 1), (4, 3, 2), (9, 5, 4), (17, 16, 1), (33, 65, 2), (130, 40, 3),
                                  (300, 9, 4), (1100, 6, 1), (5, 4, 5), (3, 17, 9), (40, 33, 21)])
def test_demag_of_random_and_uniform_states(mmlib, grid):
    nx, ny, nz = grid
    prob, oprob = make_pair(mmlib, nx, ny, nz, CELL, A=0.0, K=0.0)
    d = om.Demag(oprob)
    m = inputs.random_unit_m(oprob.shape, 900 + nx + ny + nz)
    assert rel_l2(demag(mmlib, prob, m), d.field(m)) <= 2e-15
    # saturated along each axis; the field is a small difference of large terms, so the bar is relative to Ms
    for c in range(3):
        u = np.zeros_like(m)
        u[c] = 1.0
        assert np.max(np.abs(demag(mmlib, prob, u) - d.field(u))) <= 2e-15 * 8e5


@pytest.mark.parametrize("grid", [(24, 12, 3), (10, 12, 14)])
def test_scales_exactly_with_powers_of_two(mmlib, grid):
    nx, ny, nz = grid
    prob, _ = make_pair(mmlib, nx, ny, nz, CELL, A=0.0, K=0.0)
    m = inputs.random_unit_m((nz, ny, nx), 5)
    H = demag(mmlib, prob, m)
    for e in (-200, -30, 1, 40, 300):
        assert np.array_equal(demag(mmlib, prob, np.ldexp(m, e)), np.ldexp(H, e)), e
    assert np.array_equal(demag(mmlib, prob, np.zeros_like(m)), np.zeros_like(m))
    # rows of very different magnitude share one scale downstream: each keeps its accuracy relative to the field
    m2 = m.copy()
    m2[:, :, : ny // 2] *= 2.0 ** -40
    ref = om.Demag(make_pair(mmlib, nx, ny, nz, CELL, A=0.0, K=0.0)[1]).field(m2)
    assert rel_l2(demag(mmlib, prob, m2), ref) <= 2e-15


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_inputs_come_out_as_nan(mmlib, bad):
    """A non-finite component reaches every cell of the components the tensor couples it to (for one layer H_z depends
    on m_z alone, H_x and H_y on m_x and m_y), and the minimiser reports it."""
    for nx, ny, nz in ((20, 9, 1), (20, 9, 2), (6, 5, 7)):
        prob, oprob = make_pair(mmlib, nx, ny, nz, CELL, A=0.0, K=0.0)
        m = inputs.random_unit_m(oprob.shape, 6)
        clean = demag(mmlib, prob, m)
        for c in (0, 1, 2):
            b = m.copy()
            b[c, 0, 3, 2] = bad
            H = demag(mmlib, prob, b)
            hit = {0, 1, 2} if nz > 1 else ({0, 1} if c < 2 else {2})
            for a in range(3):
                if a in hit:
                    assert np.isnan(H[a]).all()
                else:
                    # the cell's own anisotropy term mixes its components; elsewhere the field is the clean one up to
                    # rounding (the blocks' scales leave out the flagged components)
                    keep = np.ones(H[a].shape, bool)
                    keep[0, 3, 2] = False
                    assert rel_l2(H[a][keep], clean[a][keep]) <= 2e-15
        b = dev(b)
        st, _ = mmlib.mm_minimize(prob, b, (0, 0, 0), mmlib.make_opts(max_iter=5))
        assert st == mmlib.MM_ERR_NONFINITE
        assert np.array_equal(demag(mmlib, prob, m), clean)  # nothing stays behind


@pytest.mark.parametrize("prec,bar", [("MM_FP64", 2e-15), ("MM_F32X2", 2e-14)])
@pytest.mark.parametrize("grid", [(1, 9, 1), (9, 1, 2), (33, 18, 3), (200, 7, 4)])
def test_exchange_on_the_integer_copy_and_beside_it(mmlib, grid, prec, bar):
    """The whole field with exchange, anisotropy and Zeeman terms: rows of one scale (integer differences), and rows
    whose scales differ (differences of the fields themselves) next to each other.  Bars: 2^-52 and 2^-46 times a small
    multiple of the terms' root-sum-square."""
    nx, ny, nz = grid
    prob, oprob = make_pair(mmlib, nx, ny, nz, (4e-9, 3e-9, 5e-9), A=1.3e-11, K=2e4, u=(0.6, 0.0, 0.8),
                            precision=getattr(mmlib, prec))
    d = om.Demag(oprob)
    m = inputs.random_unit_m(oprob.shape, 31 + nx)
    states = [m, m * 2.0 ** -30, m * np.where(np.arange(ny) % 3 == 0, 2.0 ** -12, 1.0).reshape(1, 1, ny, 1)]
    for s in states:
        H = torch.empty(s.shape, dtype=torch.float64, device="cuda")
        Hext = np.array([3e3, -2e3, 1e3]) * np.max(np.abs(s))
        mmlib.mm_heff(prob, dev(s), Hext, H)
        assert rel_l2(H.cpu().numpy(), om.heff(oprob, s, Hext, d)) <= bar
        E = mmlib.mm_energy(prob, dev(s), Hext)
        ref = om.energy(oprob, s, Hext, d)
        keys = ["demag", "exchange", "anisotropy", "zeeman", "total"]
        scale = max(abs(ref[k]) for k in keys)
        for i, k in enumerate(keys):
            assert abs(E[i] - ref[k]) <= 1e-12 * scale, k

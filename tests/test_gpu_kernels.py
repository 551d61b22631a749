"""GPU: the kernels' size rules at their edges, against the FP64 oracle.

Tolerances (relative L2): whole steps FP64 1e-10, FP32 1e-5 on the field over
a few steps (some ten rounded operations of 6e-8 per step and value); rho of
an ionising row goes with the eighth power of the intensity, so 16 times the
field's relative error.  Row sums of a given field: 24 bits per |A|^2 in FP32,
averaged over the row, and FP64 sums.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1507_05988_gb300 import workloads as W
from tests.conftest import rel_l2

pytestmark = pytest.mark.gpu

FP64, FP32 = 0, 1
TOL = {FP64: 1e-10, FP32: 1e-5}
RHO_TOL = {FP64: 1.6e-9, FP32: 1.6e-4}


@pytest.fixture(scope="module")
def fcn():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_1507_05988_gb300 import build
    build.build()
    from paper_1507_05988_gb300 import fcn as m
    return m


def _check(fcn, wl, prec, dz, n, variants=None, rho=False):
    pb = oracle.Problem(**wl.physics())
    s = fcn.Solver(wl.physics(), precision=prec)
    if variants is not None:
        s.set_variants(*variants)
    s.set_field(wl.field())
    s.step(dz, n)
    A, r = s.get_field(), s.get_rho()
    s.close()
    Aref, rref = oracle.run(pb, dz, n, wl.field())
    assert rel_l2(A, Aref) < TOL[prec]
    if rho:
        assert rref.max() > 1e12
        assert rel_l2(r, rref) < RHO_TOL[prec]


# rows that only rotate, with and without n6 / n8, in every form of the row
# kernel; 7 rows: the last pair has one row
@pytest.mark.parametrize("nt", [256, 512, 1024, 2048, 4096, 8192])
@pytest.mark.parametrize("row_v", [0, 1, 2, 3])
@pytest.mark.parametrize("n2j", [(W.N2, W.N4, 0, 0), (W.N2, W.N4, 2e-57, -4e-73)])
def test_row_forms_with_an_odd_number_of_rows(fcn, nt, row_v, n2j):
    _check(fcn, W.small(7, nt, p_over_pcr=3.0, noise_seed=4).with_(n2j=n2j), FP32, 5e-3, 3, (row_v, 0))


# the number of rows up to which four values per thread serve a grid, and the
# next one
THIN = [(FP64, 389, 1024), (FP64, 390, 1024), (FP64, 7, 64), (FP64, 130, 128),
        (FP32, 526, 512), (FP32, 527, 512), (FP32, 7, 64), (FP32, 130, 128)]


@pytest.mark.parametrize("prec,nr,nt", THIN)
def test_small_grid_rows(fcn, prec, nr, nt):
    wl = W.small(nr, nt, p_over_pcr=5.0).with_(n2j=(W.N2, W.N4, 0, 0))
    _check(fcn, wl, prec, 1e-3, 3)


# rows that ionise: plasma phase, loss and the rho scan.  Without diffraction
# and dispersion, so that a step is the row stage alone and an error of the
# input stays of its size (with them the phase gradients of so intense a beam
# amplify it: the oracle moves by 1e-4 to 1 for 6e-8)
@pytest.mark.parametrize("prec,nr,nt,row_v",
                         [(FP32, 7, nt, v) for nt in (256, 512, 1024, 2048, 4096, 8192) for v in range(6)] +
                         [(FP64, 7, nt, 0) for nt in (256, 2048, 8192)] + [c + (0,) for c in THIN])
def test_ionising_rows(fcn, prec, nr, nt, row_v):
    wl = W.small(nr, nt, w0=0.2e-3, p_over_pcr=6.0).with_(flags=W.KERR | W.PLASMA | W.MPI)
    _check(fcn, wl, prec, 1e-4, 2, (row_v, 0), rho=True)


@pytest.mark.parametrize("prec", [FP64, FP32])
@pytest.mark.parametrize("nr", [3, 4, 7, 8, 9, 16, 17, 33, 129, 257, 1025])
@pytest.mark.parametrize("col_v", [4, 5, 6, 7])
def test_column_blocks_at_chunk_edges(fcn, prec, nr, col_v):
    _check(fcn, W.small(nr, 32, p_over_pcr=3.0, noise_seed=11), prec, 5e-3, 2, (0, col_v))


@pytest.mark.parametrize("shapes", [((256, 512), (3, 1024)), ((512, 512), (257, 2048)), ((513, 512), (9, 4096))])
def test_batched_columns_by_the_tallest_grid(fcn, shapes):
    wls = [W.small(nr, nt, p_over_pcr=2.0 + k, noise_seed=k + 1) for k, (nr, nt) in enumerate(shapes)]
    s = fcn.Solver([w.physics() for w in wls], precision=FP32)
    for i, w in enumerate(wls):
        s.set_field(w.field(), pulse=i)
    s.step(2e-3, 3)
    outs = [s.get_field(i) for i in range(len(wls))]
    s.close()
    for out, w in zip(outs, wls):
        assert rel_l2(out, oracle.run(oracle.Problem(**w.physics()), 2e-3, 3, w.field())[0]) < 1e-5, w.name


# row totals: one to 512 threads per row
@pytest.mark.parametrize("prec", [FP64, FP32])
@pytest.mark.parametrize("nt", [4, 16, 32, 64, 256, 1024, 4096, 8192])
def test_row_sums_of_the_statistics(fcn, prec, nt):
    wl = W.small(7, nt, w0=0.2e-3, p_over_pcr=6.0)
    pb = oracle.Problem(**wl.physics())
    s = fcn.Solver(wl.physics(), precision=prec)
    s.set_field(wl.field())
    s.step(1e-3, 2)
    A, rho, d = s.get_field(), s.get_rho(), s.diag()
    s.close()
    ref = oracle.diag(pb, A, rho)
    tol = 1e-12 if prec == FP64 else 2e-7
    for k in ("energy", "peak_intensity", "onaxis_peak", "peak_rho"):
        assert d[k] == pytest.approx(ref[k], rel=tol), k


@pytest.mark.parametrize("prec", [FP64, FP32])
@pytest.mark.parametrize("nt", [16, 32, 256, 2048, 4096, 8192])
def test_row_sums_of_the_step_doubling_norm(fcn, prec, nt):
    """One attempt against its own two fields: sqrt(sum |A1 - A2|^2 / sum
    |A2|^2), A1 after one step and A2 after two half steps.  In FP32 both
    differ from the attempt's by roundings of 1e-6 of the field."""
    wl = W.small(7, nt, w0=0.2e-3, p_over_pcr=6.0, noise_seed=2)
    h, out = 5e-3, []
    for n in (1, 2):
        s = fcn.Solver(wl.physics(), precision=prec)
        s.set_field(wl.field())
        s.step(h / n, n)
        out.append(s.get_field())
        s.close()
    s = fcn.Solver(wl.physics(), precision=prec)
    s.set_field(wl.field())
    st = s.propagate(h, h, rtol=1e3)
    s.close()
    assert st["substeps"] == 3
    err = rel_l2(out[0], out[1])
    assert st["last_err"] == pytest.approx(err, rel=1e-9 if prec == FP64 else 1e-4, abs=1e-12 if prec == FP64 else 1e-6)


@pytest.mark.parametrize("prec", [FP64, FP32])
@pytest.mark.parametrize("nr,nt", [(3, 16), (33, 64), (1000, 32)])
def test_power_profile(fcn, prec, nr, nt):
    wl = W.small(nr, nt, p_over_pcr=3.0, noise_seed=4)
    s = fcn.Solver(wl.physics(), precision=prec)
    s.set_field(wl.field())
    s.step(1e-3, 1)
    A, (power, fluence) = s.get_field(), s.profiles()
    s.close()
    ref = oracle.diag(oracle.Problem(**wl.physics()), A)
    tol = 1e-12 if prec == FP64 else 2e-7
    assert rel_l2(power, ref["power"]) < tol
    assert rel_l2(fluence, ref["fluence"]) < tol


# Cartesian lines: chunk edges of both axes, an odd number of lines, and no
# diffraction (the factors are the identity up to the dispersion)
@pytest.mark.parametrize("prec", [FP64, FP32])
@pytest.mark.parametrize("nx,ny", [(3, 3), (16, 17), (33, 9), (65, 31), (129, 5)])
@pytest.mark.parametrize("line_v", [0, 1, 2, 3, 4, 5, 6, 7])
def test_cartesian_lines_at_chunk_edges(fcn, prec, nx, ny, line_v):
    wl = W.small_xy(nx, ny, 16, p_over_pcr=3.0, noise_seed=5, dz=1e-2)
    for flags in (W.ALL_PHYSICS, W.ALL_PHYSICS & ~W.DIFFRACTION):
        d = dict(wl.physics(), flags=flags)
        s = fcn.SolverXY(wl.grid(), d, precision=prec)
        s.set_variants(0, line_v)
        s.set_field(wl.field())
        s.step(wl.dz, 3)
        A = s.get_field()
        s.close()
        ref, _ = oracle.xy_run(oracle.Problem(**d), oracle.GridXY(**wl.grid()), wl.dz, 3, wl.field())
        assert rel_l2(A, ref) < TOL[prec], flags

"""GPU: calls beside the usual ones (physics terms switched off, other photon
numbers, uneven contexts) that have to stay as right and as fast as those."""
import ctypes as C
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle
from paper_1507_05988_gb300 import workloads as W
from tests.conftest import ROOT, rel_l2

pytestmark = pytest.mark.gpu

FP64, FP32 = 0, 1


@pytest.fixture(scope="module")
def fcn():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_1507_05988_gb300 import build
    build.build()
    from paper_1507_05988_gb300 import fcn as m
    return m


def _best_ms(run, reps=9):
    """Shortest of reps runs between CUDA events, after two untimed ones."""
    out = []
    for i in range(reps + 2):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        e0.record()
        run()
        e1.record()
        torch.cuda.synchronize()
        out.append(e0.elapsed_time(e1))
    return min(out[2:])


def test_cartesian_step_without_diffraction_is_no_slower(fcn):
    """Without diffraction the line stage is pointwise.  Its step took four
    times that with diffraction where each thread had one load in flight; a
    factor of two leaves room for what the timing varies."""
    wl = W.small_xy(255, 31, 64, p_over_pcr=3.0, dz=1e-3)
    ms = {}
    for flags in (W.ALL_PHYSICS, W.ALL_PHYSICS & ~W.DIFFRACTION):
        s = fcn.SolverXY(wl.grid(), dict(wl.physics(), flags=flags), precision=FP32)
        s.set_field(wl.field())
        ms[flags] = _best_ms(lambda: s.step(wl.dz, 16))
        s.close()
    assert ms[W.ALL_PHYSICS & ~W.DIFFRACTION] < 2 * ms[W.ALL_PHYSICS], ms


@pytest.mark.parametrize("prec,nr,nt", [(FP32, 1024, 2048), (FP64, 1024, 256)])
def test_loss_without_plasma_does_not_scan(fcn, prec, nr, nt):
    """With loss and neither plasma nor saturation nothing reads the density:
    rows that ionise take 0.83 to 0.89 of the time with saturation, which
    needs the scan along tau (1.00 where the scan ran all the same)."""
    wl = W.small(nr, nt)
    field = np.full((nr, nt), np.sqrt(1e17), dtype=np.complex128)
    ms = {}
    for flags in (W.KERR | W.MPI, W.KERR | W.MPI | W.MPI_SAT):
        s = fcn.Solver(dict(wl.physics(), flags=flags), precision=prec)
        s.set_variants(0, 4)
        s.set_field(field)
        ms[flags] = _best_ms(lambda: s.step(1e-6, 17))
        s.close()
    assert ms[W.KERR | W.MPI] < 0.95 * ms[W.KERR | W.MPI | W.MPI_SAT], ms


@pytest.mark.parametrize("prec,bits", [(FP64, b << 32 | c) for b, c in ((0x7FF80000, 0), (0x7FFFFFFF, 0xFFFFFFFF),
                                                                        (0xFFFFFFFF, 0xFFFFFFFF), (0x7FF00000, 0))] +
                         [(FP32, b) for b in (0x7FC00000, 0x7FFFFFFF, 0xFFFFFFFF, 0x7F800000)])
def test_a_row_that_is_not_finite_leaves_its_neighbours_alone(fcn, prec, bits):
    """The rows of one CTA share the bound that picks their half step's form.
    A NaN or infinity in one, whatever its bits, changes no other row (equal
    forms: to some roundings, 1e-14 and 1e-6)."""
    wl = W.small(8, 256, p_over_pcr=3.0, noise_seed=2)
    g, p = fcn.grid_params(wl.physics())
    out = []
    for bad in (False, True):
        f = wl.field().astype(np.complex128 if prec == FP64 else np.complex64)
        if bad:
            f.view(np.uint64 if prec == FP64 else np.uint32)[1, 14] = bits
        f = torch.from_numpy(f).cuda()
        assert fcn.fcn_op_rows(C.byref(g), C.byref(p), prec, fcn.FCN_OP_NL, 1e-2, fcn.tensor_ptr(f), None,
                               fcn.stream_ptr()) == 0
        torch.cuda.synchronize()
        out.append(f.cpu().numpy().astype(np.complex128))
    keep = [r for r in range(wl.nr) if r != 1]
    ref, res = out[0][keep], out[1][keep]
    assert np.linalg.norm(ref - wl.field()[keep]) > 1e-4 * np.linalg.norm(ref)        # the half step acts
    assert np.linalg.norm(res - ref) < (1e-14 if prec == FP64 else 1e-6) * np.linalg.norm(ref)


_TUNE_RUN = """
from paper_1507_05988_gb300 import fcn, workloads as W
wl = W.small(64, 256)
for K in (7, 8, 8):
    s = fcn.Solver(dict(wl.physics(), K=K), precision=fcn.FCN_FP32_MIXED)
    s.set_field(wl.field())
    s.step(1e-3, 2)
    s.close()
"""


def test_variant_choices_by_photon_number_and_format(fcn, tmp_path):
    """The row variants serve K = 8 only: another K's choice (variant 0,
    untimed) is not a K = 8 context's.  Lines of an older format, whose numbers
    meant other kernels, are passed over, and this format's are read back."""
    path = tmp_path / "variants"
    path.write_text("1 64 256 5 3\n")
    for _ in range(2):
        subprocess.run([sys.executable, "-c", _TUNE_RUN], check=True, cwd=ROOT, timeout=300,
                       env=dict(os.environ, FCN_TUNE_CACHE=str(path)))
        lines = path.read_text().splitlines()
        assert lines[0] == "1 64 256 5 3" and len(lines) == 3
        fmt = {ln.split()[0] for ln in lines[1:]}
        assert len(fmt) == 1 and not fmt.pop().isdigit()
        assert [ln.split()[1:5] for ln in lines[1:]] == [["1", "64", "256", "0"], ["1", "64", "256", "1"]]


# both sides of the line between work lists and launches per pulse, pulses of
# like size whose tall one would leave the other's column CTAs half empty, and
# many small pulses beside a tall one
@pytest.mark.parametrize("shapes,lists", [(((195, 2048), (390, 1024)), True), (((585, 2048), (1171, 1024)), False),
                                          (((97, 8192), (195, 4096)), True), (((195, 4096), (1562, 512)), False),
                                          (((128, 512),) * 40 + ((2048, 1024),), True)])
def test_work_lists_by_the_size_of_the_pulses(fcn, shapes, lists):
    s = fcn.Solver([W.small(nr, nt).physics() for nr, nt in shapes], precision=FP32)
    for i, (nr, nt) in enumerate(shapes):
        s.set_field(np.zeros((nr, nt), np.complex128), pulse=i)
    s.step(1e-3, 1)
    s.profile(True)
    s.profile_read()
    s.step(1e-3, 1)
    n = s.profile_read()
    s.close()
    assert [n[k][1] for k in ("row_head", "column", "row_tail")] == [1 if lists else len(shapes)] * 3


@pytest.mark.parametrize("shapes", [((256, 512), (3, 1024)), ((512, 512), (257, 2048)), ((513, 512), (9, 4096))])
def test_forced_work_lists(fcn, shapes):
    """Column CTAs of each size, whatever the automatic choice: 1e-5 after
    three steps, as for the launches per pulse."""
    wls = [W.small(nr, nt, p_over_pcr=2.0 + k, noise_seed=k + 1) for k, (nr, nt) in enumerate(shapes)]
    s = fcn.Solver([w.physics() for w in wls], precision=FP32)
    s.set_batching(1)
    for i, w in enumerate(wls):
        s.set_field(w.field(), pulse=i)
    s.step(2e-3, 3)
    outs = [s.get_field(i) for i in range(len(wls))]
    s.close()
    for out, w in zip(outs, wls):
        assert rel_l2(out, oracle.run(oracle.Problem(**w.physics()), 2e-3, 3, w.field())[0]) < 1e-5, w.name

"""GPU parity of the Poisson and Helmholtz solves against the FP64 oracle.

Every case builds a seeded synthetic right-hand side, runs the CUDA path
through the C ABI and compares element by element with the oracle
(relative L2).  Shapes cover the one-CTA-per-plane transform path, the
split x/z path (planes larger than shared memory), radix-3 sizes, ragged
pencil tiles and the smallest supported grid.
"""

import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

from oracle import ibm_oracle as O
from paper_2406_19920_gb300 import synth
import paper_2406_19920_gb300 as ibm
from tests.gpu_util import TOL_FP32, TOL_FP64, dev, grid, host, rel_err, solve_extended

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPES = [
    (32, 32, 32),     # workload-0 grid, plane path
    (8, 8, 8),        # smallest grid
    (12, 10, 24),     # radix 3, odd ny, ragged pencil tile
    (48, 40, 48),     # radix 3
    (96, 33, 64),     # mixed shape, odd ny
    (256, 12, 256),   # plane larger than shared memory (split x/z path)
    (384, 9, 32),     # longest radix-3 row, split path
    (16, 200, 24),    # pencils of 200: FP32 split-component block solve, FP64 serial sweep
    (32, 300, 16),    # pencils longer than 256: serial sweep in both precisions
]


def _plan(nx, ny, nz, g, prec, refine=1):
    return ibm.ibm_plan_create(nx, ny, nz, g[3:], prec, refine)


@pytest.mark.parametrize("shape", SHAPES)
def test_poisson_fp64_matches_oracle(shape):
    nx, ny, nz = shape
    g = grid(nx, ny, nz)
    b = synth.white_noise(nx, ny, nz, workload=10, stream=0) + 0.3
    ref, mean_b = O.poisson_solve(b, g)
    plan = _plan(nx, ny, nz, g, ibm.IBM_FP64)
    try:
        rhs = dev(b, torch.float64)
        phi = torch.empty_like(rhs)
        info = ibm.ibm_poisson_solve(plan, rhs, phi, info=True)
        assert rel_err(host(phi), ref) <= TOL_FP64
        assert abs(info["removed_mean"] - mean_b) <= 1e-12 * max(1.0, abs(mean_b))
        assert info["rel_residual"] < 1e-12
    finally:
        ibm.ibm_plan_destroy(plan)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("refine", [1, 2])
def test_poisson_fp32_refined_matches_oracle(shape, refine):
    nx, ny, nz = shape
    g = grid(nx, ny, nz)
    b32 = synth.white_noise(nx, ny, nz, workload=11, stream=0).astype(np.float32)
    ref, _ = O.poisson_solve(b32.astype(np.float64), g)
    plan = _plan(nx, ny, nz, g, ibm.IBM_FP32_REFINED, refine)
    try:
        rhs = dev(b32, torch.float32)
        phi = torch.empty_like(rhs)
        info = ibm.ibm_poisson_solve(plan, rhs, phi, info=True)
        assert rel_err(host(phi), ref) <= TOL_FP32
        assert info["refine_iters"] == refine
    finally:
        ibm.ibm_plan_destroy(plan)


def test_poisson_workload0_eigen_rhs_both_precisions():
    """Workload 0: 32^3, sum of 4 grid eigenfunctions + noise 1e-3."""
    g = grid(32, 32, 32)
    b, _ = synth.rhs_eigen_sum(32, 32, 32, workload=0)
    for prec, dt, tol in ((ibm.IBM_FP64, torch.float64, TOL_FP64), (ibm.IBM_FP32_REFINED, torch.float32, TOL_FP32)):
        bb = b.astype(np.float32).astype(np.float64) if dt == torch.float32 else b
        ref, _ = O.poisson_solve(bb, g)
        plan = _plan(32, 32, 32, g, prec)
        try:
            rhs = dev(bb, dt)
            phi = torch.empty_like(rhs)
            ibm.ibm_poisson_solve(plan, rhs, phi)
            torch.cuda.synchronize()
            assert rel_err(host(phi), ref) <= tol
        finally:
            ibm.ibm_plan_destroy(plan)


def test_poisson_in_place_and_128_lowpass():
    """Workload 1 right-hand side (128^3 low-passed noise), rhs == phi."""
    g = grid(128, 128, 128)
    b = synth.rhs_lowpass_noise(128, 128, 128, kmax=32.0, workload=1).astype(np.float32)
    ref, _ = O.poisson_solve(b.astype(np.float64), g)
    plan = _plan(128, 128, 128, g, ibm.IBM_FP32_REFINED, 1)
    try:
        x = dev(b, torch.float32)
        info = ibm.ibm_poisson_solve(plan, x, x, info=True)
        err = rel_err(host(x), ref)
        assert err <= TOL_FP32, (err, info)
    finally:
        ibm.ibm_plan_destroy(plan)


@pytest.mark.parametrize("shape", [(32, 32, 32), (12, 10, 24), (256, 12, 256), (48, 17, 96), (24, 129, 16)])
@pytest.mark.parametrize("bc", [ibm.IBM_FIELD_CELL_NEUMANN, ibm.IBM_FIELD_CELL_DIRICHLET,
                                ibm.IBM_FIELD_FACE_DIRICHLET])
@pytest.mark.parametrize("c", [5e-6, 0.05])
def test_helmholtz_matches_oracle(shape, bc, c):
    nx, ny, nz = shape
    g = grid(nx, ny, nz)
    r = synth.white_noise(nx, ny, nz, workload=12, stream=bc)
    for prec, dt, tol in ((ibm.IBM_FP64, torch.float64, TOL_FP64), (ibm.IBM_FP32_REFINED, torch.float32, TOL_FP32)):
        rr = r.astype(np.float32).astype(np.float64) if dt == torch.float32 else r
        ref = O.helmholtz_solve(rr, g, c, bc)
        plan = _plan(nx, ny, nz, g, prec, 1)
        try:
            rhs = dev(rr, dt)
            u = torch.empty_like(rhs)
            ibm.ibm_helmholtz_solve(plan, c, bc, rhs, u)
            torch.cuda.synchronize()
            got = host(u)
            assert rel_err(got, ref) <= tol, (prec, rel_err(got, ref))
            if bc == ibm.IBM_FIELD_FACE_DIRICHLET:
                assert np.all(got[0] == 0.0)
        finally:
            ibm.ibm_plan_destroy(plan)


# Planes with a cluster transform (C CTAs per plane exchanging rows and
# columns through distributed shared memory), each solved in every plane
# mode the shape has: 0 split x/z passes, 1 one CTA per plane, 2/4/8 cluster.
PLANE_MODE_SHAPES = [
    (64, 10, 64), (96, 9, 96), (128, 12, 128), (192, 8, 192), (256, 9, 256),
    (384, 8, 256), (256, 8, 128), (128, 8, 256), (384, 8, 384), (512, 8, 256),
]


def _plan_in_mode(nx, ny, nz, g, prec, refine, mode):
    os.environ["IBM_PLANE_MODE"] = str(mode)
    try:
        return ibm.ibm_plan_create(nx, ny, nz, g[3:], prec, refine)
    except ibm.IbmError as e:
        assert e.code == ibm.IBM_ERR_UNSUPPORTED
        return None
    finally:
        del os.environ["IBM_PLANE_MODE"]


@pytest.mark.parametrize("shape", PLANE_MODE_SHAPES)
def test_every_plane_mode_matches_oracle(shape):
    nx, ny, nz = shape
    g = grid(nx, ny, nz)
    b = synth.white_noise(nx, ny, nz, workload=13, stream=0) + 0.2
    b32 = b.astype(np.float32).astype(np.float64)
    ref64, _ = O.poisson_solve(b, g)
    ref32, _ = O.poisson_solve(b32, g)
    href = O.helmholtz_solve(b32, g, 0.01, ibm.IBM_FIELD_CELL_DIRICHLET)
    ran = set()
    for mode in (0, 1, 2, 4, 8):
        for prec, dt, tol, bb, ref in ((ibm.IBM_FP64, torch.float64, TOL_FP64, b, ref64),
                                       (ibm.IBM_FP32_REFINED, torch.float32, TOL_FP32, b32, ref32)):
            plan = _plan_in_mode(nx, ny, nz, g, prec, 1, mode)
            if plan is None:
                continue
            ran.add(mode)
            try:
                rhs = dev(bb, dt)
                phi = torch.empty_like(rhs)
                ibm.ibm_poisson_solve(plan, rhs, phi)
                torch.cuda.synchronize()
                assert rel_err(host(phi), ref) <= tol, (mode, prec, rel_err(host(phi), ref))
                if prec == ibm.IBM_FP32_REFINED:
                    u = torch.empty_like(rhs)
                    ibm.ibm_helmholtz_solve(plan, 0.01, ibm.IBM_FIELD_CELL_DIRICHLET, rhs, u)
                    torch.cuda.synchronize()
                    assert rel_err(host(u), href) <= tol, (mode, rel_err(host(u), href))
                ibm.ibm_plan_check(plan)
            finally:
                ibm.ibm_plan_destroy(plan)
    assert 0 in ran and any(m >= 2 for m in ran), ran


PENCIL_MODE_SHAPES = [(32, 32, 32), (12, 10, 24), (48, 17, 96), (24, 129, 16), (16, 200, 24), (32, 300, 16)]


@pytest.mark.parametrize("shape", PENCIL_MODE_SHAPES)
def test_every_pencil_kernel_matches_oracle(shape):
    """IBM_PENCIL_MODE 1 (warp-parallel blocks), 2 (tile sweep), 3 (streaming sweep), 4 (segmented sweep)."""
    nx, ny, nz = shape
    g = grid(nx, ny, nz)
    b = synth.white_noise(nx, ny, nz, workload=14, stream=0) + 0.1
    b32 = b.astype(np.float32).astype(np.float64)
    ref64, _ = O.poisson_solve(b, g)
    ref32, _ = O.poisson_solve(b32, g)
    helm = {bc: O.helmholtz_solve(b32, g, 0.02, bc)
            for bc in (ibm.IBM_FIELD_CELL_NEUMANN, ibm.IBM_FIELD_FACE_DIRICHLET)}
    for mode in (1, 2, 3, 4):
        for prec, dt, tol, bb, ref in ((ibm.IBM_FP64, torch.float64, TOL_FP64, b, ref64),
                                       (ibm.IBM_FP32_REFINED, torch.float32, TOL_FP32, b32, ref32)):
            os.environ["IBM_PENCIL_MODE"] = str(mode)
            try:
                plan = ibm.ibm_plan_create(nx, ny, nz, g[3:], prec, 1)
            finally:
                del os.environ["IBM_PENCIL_MODE"]
            try:
                rhs = dev(bb, dt)
                phi = torch.empty_like(rhs)
                ibm.ibm_poisson_solve(plan, rhs, phi)
                torch.cuda.synchronize()
                assert rel_err(host(phi), ref) <= tol, (mode, prec, rel_err(host(phi), ref))
                if prec == ibm.IBM_FP32_REFINED:
                    for bc, href in helm.items():
                        u = torch.empty_like(rhs)
                        ibm.ibm_helmholtz_solve(plan, 0.02, bc, rhs, u)
                        torch.cuda.synchronize()
                        assert rel_err(host(u), href) <= tol, (mode, bc, rel_err(host(u), href))
                ibm.ibm_plan_check(plan)
            finally:
                ibm.ibm_plan_destroy(plan)


@pytest.mark.parametrize("shape", [(32, 256, 32), (16, 500, 16), (24, 129, 16)])
def test_segmented_sweep_unrefined_fp32_accuracy(shape):
    """Without refinement the FP32 error is the sweep's own: the segmented
    sweep (pivot prefix, carries combined across warps) stays within a small
    factor of the single two-ended sweep on long, near-singular pencils."""
    nx, ny, nz = shape
    g = grid(nx, ny, nz)
    b32 = synth.white_noise(nx, ny, nz, workload=15, stream=0).astype(np.float32)
    ref, _ = O.poisson_solve(b32.astype(np.float64), g)
    errs = {}
    for mode in (3, 4):
        os.environ["IBM_PENCIL_MODE"] = str(mode)
        try:
            plan = ibm.ibm_plan_create(nx, ny, nz, g[3:], ibm.IBM_FP32_REFINED, 0)
        finally:
            del os.environ["IBM_PENCIL_MODE"]
        try:
            rhs = dev(b32, torch.float32)
            phi = torch.empty_like(rhs)
            ibm.ibm_poisson_solve(plan, rhs, phi)
            torch.cuda.synchronize()
            errs[mode] = rel_err(host(phi), ref)
        finally:
            ibm.ibm_plan_destroy(plan)
    assert errs[4] <= 1e-5, errs
    assert errs[4] <= 2.0 * errs[3] + 1e-7, errs


def test_fp32_fields_must_be_16_byte_aligned():
    """The four-point residual and the vector loads need 16-byte aligned
    fields: an element-aligned view at an odd offset is refused before any
    launch, the aligned view of the same buffer solves."""
    nx, ny, nz = 32, 24, 16
    g = grid(nx, ny, nz)
    n = nx * ny * nz
    b32 = synth.white_noise(nx, ny, nz, workload=16, stream=0).astype(np.float32)
    ref, _ = O.poisson_solve(b32.astype(np.float64), g)
    plan = _plan(nx, ny, nz, g, ibm.IBM_FP32_REFINED, 2)
    try:
        buf = torch.zeros(n + 4, dtype=torch.float32, device="cuda")
        out = torch.zeros(n + 4, dtype=torch.float32, device="cuda")
        for off in (1, 3):
            with pytest.raises(ibm.IbmError) as e:
                ibm.ibm_poisson_solve(plan, buf[off:off + n].view(ny, nz, nx), out[off:off + n].view(ny, nz, nx))
            assert e.value.code == ibm.IBM_ERR_ARG
        rhs = buf[4:4 + n].view(ny, nz, nx)
        rhs.copy_(dev(b32, torch.float32))
        phi = out[4:4 + n].view(ny, nz, nx)
        ibm.ibm_poisson_solve(plan, rhs, phi)
        torch.cuda.synchronize()
        assert rel_err(host(phi), ref) <= TOL_FP32
    finally:
        ibm.ibm_plan_destroy(plan)


@pytest.mark.parametrize("prec", [ibm.IBM_FP64, ibm.IBM_FP32_REFINED])
@pytest.mark.parametrize("shape", [(32, 24, 16), (48, 17, 96)])
def test_solves_with_wall_data_match_oracle(prec, shape):
    """Inhomogeneous wall data (Appendix B's boundary right-hand sides, BC2.2):
    Poisson with dphi/dy on both walls and Helmholtz with wall values / wall
    slopes for every field kind, against the oracle; rhs left untouched."""
    nx, ny, nz = shape
    g = grid(nx, ny, nz)
    dt = torch.float64 if prec == ibm.IBM_FP64 else torch.float32
    npdt = np.float64 if prec == ibm.IBM_FP64 else np.float32
    tol = TOL_FP64 if prec == ibm.IBM_FP64 else TOL_FP32
    rng = np.random.default_rng(nx + ny)
    b = synth.white_noise(nx, ny, nz, workload=17, stream=0).astype(npdt).astype(np.float64)
    lo, hi = (rng.standard_normal((nz, nx)).astype(npdt).astype(np.float64) for _ in range(2))
    plan = ibm.ibm_plan_create(nx, ny, nz, g[3:], prec, 1)
    try:
        rhs, glo, ghi = dev(b, dt), dev(lo, dt), dev(hi, dt)
        keep = rhs.clone()
        phi = torch.empty_like(rhs)
        info = ibm.ibm_poisson_solve_bc(plan, rhs, phi, glo, ghi, info=True)
        ref, removed = O.poisson_solve(b, g, q_lo=lo, q_hi=hi)
        assert rel_err(host(phi), ref) <= tol
        assert abs(info["removed_mean"] - removed) <= 1e-5 * max(1.0, abs(removed))
        for bc in (ibm.IBM_FIELD_CELL_NEUMANN, ibm.IBM_FIELD_CELL_DIRICHLET, ibm.IBM_FIELD_FACE_DIRICHLET):
            u = torch.empty_like(rhs)
            ibm.ibm_helmholtz_solve_bc(plan, 0.02, bc, rhs, u, glo, ghi)
            torch.cuda.synchronize()
            href = O.helmholtz_solve(b, g, 0.02, bc, lo, hi)
            assert rel_err(host(u), href) <= tol, bc
            # one wall only
            ibm.ibm_helmholtz_solve_bc(plan, 0.02, bc, rhs, u, None, ghi)
            torch.cuda.synchronize()
            assert rel_err(host(u), O.helmholtz_solve(b, g, 0.02, bc, None, hi)) <= tol, bc
        assert torch.equal(rhs, keep)
        # in place
        ibm.ibm_helmholtz_solve_bc(plan, 0.02, ibm.IBM_FIELD_CELL_DIRICHLET, rhs, rhs, glo, ghi)
        torch.cuda.synchronize()
        assert rel_err(host(rhs), O.helmholtz_solve(b, g, 0.02, ibm.IBM_FIELD_CELL_DIRICHLET, lo, hi)) <= tol
        ibm.ibm_plan_check(plan)
    finally:
        ibm.ibm_plan_destroy(plan)


def test_wall_data_rejected_without_walls():
    g = grid(16, 16, 16)
    plan = ibm.ibm_plan_create(16, 16, 16, g[3:], ibm.IBM_FP64, 0, bc=ibm.IBM_BC_TRIPLY_PERIODIC)
    try:
        x = torch.zeros((16, 16, 16), dtype=torch.float64, device="cuda")
        with pytest.raises(ibm.IbmError) as e:
            ibm.ibm_poisson_solve_bc(plan, x, x, x[0], x[0])
        assert e.value.code == ibm.IBM_ERR_UNSUPPORTED
        with pytest.raises(ibm.IbmError) as e:
            ibm.ibm_helmholtz_solve_bc(plan, 0.1, ibm.IBM_FIELD_CELL_NEUMANN, x, x, x[0], x[0])
        assert e.value.code == ibm.IBM_ERR_UNSUPPORTED
    finally:
        ibm.ibm_plan_destroy(plan)


def test_invalid_arguments_rejected_before_launch():
    g = grid(32, 32, 32)
    with pytest.raises(ibm.IbmError) as e:
        ibm.ibm_plan_create(30, 32, 32, g[3:], ibm.IBM_FP32_REFINED, 1)
    assert e.value.code == ibm.IBM_ERR_ARG
    with pytest.raises(ibm.IbmError):
        ibm.ibm_plan_create(32, 4, 32, g[3:], ibm.IBM_FP32_REFINED, 1)
    with pytest.raises(ibm.IbmError):
        ibm.ibm_plan_create(32, 32, 32, (1.0, -1.0, 1.0), ibm.IBM_FP64, 0)
    plan = _plan(32, 32, 32, g, ibm.IBM_FP64)
    try:
        x = torch.zeros(32 * 32 * 32 + 1, dtype=torch.float64, device="cuda")
        with pytest.raises(ibm.IbmError):
            ibm.ibm_poisson_solve(plan, x[1:].data_ptr() + 4, x.data_ptr())
        with pytest.raises(ibm.IbmError):
            ibm.ibm_helmholtz_solve(plan, -1.0, 0, x, x)
    finally:
        ibm.ibm_plan_destroy(plan)


@pytest.mark.parametrize("prec", [ibm.IBM_FP64, ibm.IBM_FP32_REFINED])
@pytest.mark.parametrize("n", [8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512])
def test_split_rows_every_length_last_cta_partial(n, prec, monkeypatch):
    """x rows and z columns of every length through the split passes (9 planes
    of 12 or n rows: the row pairs and the columns do not fill the last CTA)."""
    monkeypatch.setenv("IBM_PLANE_MODE", "0")
    dt, tol = (torch.float64, TOL_FP64) if prec == ibm.IBM_FP64 else (torch.float32, TOL_FP32)
    for nx, nz in ((n, 12), (12, n)):
        g = grid(nx, 9, nz)
        b = synth.white_noise(nx, 9, nz, workload=15, stream=n).astype(np.float32).astype(np.float64) + 0.25
        ref, mean_b = O.poisson_solve(b, g)
        plan = _plan(nx, 9, nz, g, prec)
        try:
            rhs = dev(b, dt)
            phi = torch.empty_like(rhs)
            info = ibm.ibm_poisson_solve(plan, rhs, phi, info=True)
            assert rel_err(host(phi), ref) <= tol
            assert abs(info["removed_mean"] - mean_b) <= (1e-12 if prec == ibm.IBM_FP64 else 1e-6)
        finally:
            ibm.ibm_plan_destroy(plan)


@pytest.mark.parametrize("mode", [2, 3])
@pytest.mark.parametrize("ny", [8, 9, 17, 33, 64, 129, 511])
def test_fp64_sweeps_constant_from_the_converged_row(ny, mode, monkeypatch):
    """The two-ended FP64 sweeps go on with constant pivots once the warp's
    pencils have converged: at once (small c), within the rows, late or never
    (Poisson, large c), over the three wall kinds and the smallest halves,
    against extended precision.  Tolerance: the terms of the excess form are all
    positive, so a half sweep of ny / 2 rows multiplies a relative error of at
    most 5 roundings (of 2^-53) a row into x, and the transforms some 40 more."""
    monkeypatch.setenv("IBM_PENCIL_MODE", str(mode))
    g = grid(24, ny, 12)
    b = synth.white_noise(24, ny, 12, workload=16, stream=ny)
    tol = (5 * ny / 2 + 40) * 2.0 ** -53
    plan = _plan(24, ny, 12, g, ibm.IBM_FP64)
    try:
        rhs = dev(b, torch.float64)
        x = torch.empty_like(rhs)
        ibm.ibm_poisson_solve(plan, rhs, x)
        err = [rel_err(host(x), solve_extended(b, g[3:]))]
        for c in (5e-6, 1e-3, 50.0):
            for bc in (O.NEUMANN, O.CELL_DIRICHLET, O.FACE_DIRICHLET):
                bb = b.copy()
                if bc == O.FACE_DIRICHLET:
                    bb[0] = 0.0
                ibm.ibm_helmholtz_solve(plan, c, bc, dev(bb, torch.float64), x)
                err.append(rel_err(host(x), solve_extended(bb, g[3:], c, bc)))
        assert max(err) <= tol, err
    finally:
        ibm.ibm_plan_destroy(plan)


@pytest.mark.parametrize("ny", [129, 144, 145, 255, 256])
@pytest.mark.parametrize("c", [2e-6, 1e-4, 5.0])
def test_fp32_segments_of_129_to_256_rows(ny, c):
    """FP32 pencils of 129 to 256 rows take 16-row segments where their pivots
    converge within one (small c) and 32-row segments otherwise; whole and
    partial last segments, the three wall kinds, beside the Poisson solve."""
    g = grid(32, ny, 24)
    b = synth.white_noise(32, ny, 24, workload=17, stream=ny).astype(np.float32).astype(np.float64)
    plan = _plan(32, ny, 24, g, ibm.IBM_FP32_REFINED)
    try:
        x = torch.empty(b.shape, dtype=torch.float32, device="cuda")
        ibm.ibm_poisson_solve(plan, dev(b, torch.float32), x)
        assert rel_err(host(x), O.poisson_solve(b, g)[0]) <= TOL_FP32
        for bc in (O.NEUMANN, O.CELL_DIRICHLET, O.FACE_DIRICHLET):
            bb = b.copy()
            if bc == O.FACE_DIRICHLET:
                bb[0] = 0.0
            ibm.ibm_helmholtz_solve(plan, c, bc, dev(bb, torch.float32), x)
            assert rel_err(host(x), O.helmholtz_solve(bb, g, c, bc)) <= TOL_FP32, bc
    finally:
        ibm.ibm_plan_destroy(plan)


@pytest.mark.parametrize("ny", [8, 31, 65, 257])
@pytest.mark.parametrize("bc", [O.NEUMANN, O.CELL_DIRICHLET, O.FACE_DIRICHLET])
def test_residual_pass_marches_every_plane(ny, bc, monkeypatch):
    """The FP32 residual pass of the split passes marches chunks of y planes:
    refined solves with one chunk a plane up to long chunks and a short last
    one, every wall kind."""
    monkeypatch.setenv("IBM_PLANE_MODE", "0")
    g = grid(128, ny, 96)
    b = synth.white_noise(128, ny, 96, workload=18, stream=ny).astype(np.float32).astype(np.float64)
    if bc == O.FACE_DIRICHLET:
        b[0] = 0.0
    plan = _plan(128, ny, 96, g, ibm.IBM_FP32_REFINED)
    try:
        x = torch.empty(b.shape, dtype=torch.float32, device="cuda")
        info = ibm.ibm_helmholtz_solve(plan, 0.01, bc, dev(b, torch.float32), x, info=True)
        assert rel_err(host(x), O.helmholtz_solve(b, g, 0.01, bc)) <= TOL_FP32
        assert info["rel_residual"] < 1e-3
    finally:
        ibm.ibm_plan_destroy(plan)


@pytest.mark.parametrize("shape", [(128, 17, 128), (128, 9, 8), (8, 9, 128), (96, 9, 128), (128, 9, 96), (12, 10, 96),
                                   (192, 9, 96), (512, 8, 16), (16, 8, 384)])
def test_plane_kernels_with_residual_inside(shape, monkeypatch):
    """FP32 plane kernels, in place up to 128 x 128 and with separate buffers
    beyond: the refined Poisson solve and the three wall kinds, whose residual
    is formed inside the forward transform."""
    monkeypatch.setenv("IBM_PLANE_MODE", "1")
    nx, ny, nz = shape
    g = grid(nx, ny, nz)
    b = synth.white_noise(nx, ny, nz, workload=19, stream=nx).astype(np.float32).astype(np.float64) + 0.25
    plan = _plan(nx, ny, nz, g, ibm.IBM_FP32_REFINED, 2)
    try:
        x = torch.empty(b.shape, dtype=torch.float32, device="cuda")
        ibm.ibm_poisson_solve(plan, dev(b, torch.float32), x)
        assert rel_err(host(x), O.poisson_solve(b, g)[0]) <= TOL_FP32
        for bc in (O.NEUMANN, O.CELL_DIRICHLET, O.FACE_DIRICHLET):
            bb = b.copy()
            if bc == O.FACE_DIRICHLET:
                bb[0] = 0.0
            ibm.ibm_helmholtz_solve(plan, 0.01, bc, dev(bb, torch.float32), x)
            assert rel_err(host(x), O.helmholtz_solve(bb, g, 0.01, bc)) <= TOL_FP32, bc
    finally:
        ibm.ibm_plan_destroy(plan)


@pytest.mark.parametrize("ny", [65, 257])
def test_poisson_residual_pass_marches_every_plane(ny, monkeypatch):
    """The same pass without the sigma term (the Poisson operator), its removed
    mean taken off b on the way: chunks of several planes and a short last one."""
    monkeypatch.setenv("IBM_PLANE_MODE", "0")
    g = grid(128, ny, 96)
    b = synth.white_noise(128, ny, 96, workload=20, stream=ny).astype(np.float32).astype(np.float64) + 0.25
    plan = _plan(128, ny, 96, g, ibm.IBM_FP32_REFINED)
    try:
        x = torch.empty(b.shape, dtype=torch.float32, device="cuda")
        ibm.ibm_poisson_solve(plan, dev(b, torch.float32), x)
        assert rel_err(host(x), O.poisson_solve(b, g)[0]) <= TOL_FP32
    finally:
        ibm.ibm_plan_destroy(plan)


def _compiled(tmp_path, name, source):
    """run() of a small program built against the library's headers."""
    from paper_2406_19920_gb300 import build as B
    src, lib = tmp_path / (name + ".cu"), tmp_path / (name + ".so")
    src.write_text(source)
    subprocess.run([B._nvcc()] + B._flags() + ["-shared", str(src), "-o", str(lib)], check=True)
    return ctypes.CDLL(str(lib)).run


RCP_CU = r"""
#include "seg.cuh"
__global__ void k(const double *x, double *r, double *d, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) { r[i] = ibm::rcp<double>(x[i]); d[i] = 1.0 / x[i]; }
}
extern "C" int run(const double *x, double *r, double *d, int n) {
  k<<<(n + 255) / 256, 256>>>(x, r, d, n);
  const cudaError_t e = cudaDeviceSynchronize();
  return (int)e;
}
"""


def test_fp64_reciprocal_within_one_unit(tmp_path):
    """The sweeps' FP64 reciprocal against 1.0 / x: at most one unit in the last
    place apart, over random mantissas with exponents of +-300, powers of two
    and their neighbours, and values next to one."""
    run = _compiled(tmp_path, "rcp", RCP_CU)
    r = np.random.default_rng(21)
    n = 1 << 22
    p = 2.0 ** np.arange(-300, 301)
    near = 1.0 + np.arange(-4096, 4097) * 2.0 ** -52
    x = np.concatenate([(1.0 + r.random(n)) * 2.0 ** r.integers(-300, 301, n), p, np.nextafter(p, np.inf),
                        np.nextafter(p, 0.0), near])
    xd = dev(x, torch.float64)
    got, div = torch.empty_like(xd), torch.empty_like(xd)
    run.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int]
    assert run(xd.data_ptr(), got.data_ptr(), div.data_ptr(), len(x)) == 0
    g, d = host(got), host(div)
    assert np.array_equal(d, 1.0 / x)
    units = np.abs(g.view(np.int64) - d.view(np.int64))
    assert units.max() <= 1, (units.max(), x[units.argmax()])
    assert (units > 0).mean() < 1e-3


DFT_CU = r"""
#include "fft2.cuh"
using namespace ibm;
// rotations first, then the plain butterflies
template <bool INV, int M, typename C> __device__ void rotated_first(C *v) {
  constexpr int N = 4 * M;
  C y[N];
  static_for<0, 4>([&](auto i1) {
    constexpr int n1 = decltype(i1)::value;
    C t[M];
    for (int n2 = 0; n2 < M; ++n2) t[n2] = v[n1 + 4 * n2];
    reg_dft<INV, M>(t);
    static_for<0, M>([&](auto i2) {
      constexpr int k2 = decltype(i2)::value;
      y[n1 * M + k2] = twiddle_const<INV, n1 * k2, N>(t[k2]);
    });
  });
  for (int k2 = 0; k2 < M; ++k2) {
    dft4<INV>(y[k2], y[M + k2], y[2 * M + k2], y[3 * M + k2]);
    for (int k1 = 0; k1 < 4; ++k1) v[k2 + M * k1] = y[k1 * M + k2];
  }
}
template <typename T, bool INV, int N> __global__ void k(const cplx<T> *x, cplx<T> *a, cplx<T> *b, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  cplx<T> u[N], w[N];
  for (int q = 0; q < N; ++q) u[q] = w[q] = x[i * N + q];
  reg_dft<INV, N>(u);
  rotated_first<INV, N / 4>(w);
  for (int q = 0; q < N; ++q) { a[i * N + q] = u[q]; b[i * N + q] = w[q]; }
}
template <typename T, int N> void go(int inv, const void *x, void *a, void *b, int n) {
  const int g = (n + 127) / 128;
  if (inv) k<T, true, N><<<g, 128>>>((const cplx<T> *)x, (cplx<T> *)a, (cplx<T> *)b, n);
  else k<T, false, N><<<g, 128>>>((const cplx<T> *)x, (cplx<T> *)a, (cplx<T> *)b, n);
}
extern "C" int run(int fp64, int len, int inv, const void *x, void *a, void *b, int n) {
  if (fp64) { len == 12 ? go<double, 12>(inv, x, a, b, n) : len == 16 ? go<double, 16>(inv, x, a, b, n) : go<double, 32>(inv, x, a, b, n); }
  else { len == 12 ? go<float, 12>(inv, x, a, b, n) : len == 16 ? go<float, 16>(inv, x, a, b, n) : go<float, 32>(inv, x, a, b, n); }
  return (int)cudaDeviceSynchronize();
}
"""


def test_folded_rotations_round_no_worse(tmp_path):
    """The register DFTs with their rotations' factors folded into the butterflies
    (12, 16 and 32 points) against rotating first, in either precision and
    direction: no larger error over 5,000 random DFTs (some 1e5 values, whose mean
    square is then known to 0.5 %), measured in the next wider precision."""
    run = _compiled(tmp_path, "dft", DFT_CU)
    run.argtypes = [ctypes.c_int] * 3 + [ctypes.c_void_p] * 3 + [ctypes.c_int]
    n = 5000
    for n_pts in (12, 16, 32):
        m = np.outer(np.arange(n_pts), np.arange(n_pts)) % n_pts
        for fp64 in (0, 1):
            wide = np.longdouble if fp64 else np.float64
            turn = 8 * np.arctan(wide(1)) * m.astype(wide) / n_pts
            x = np.random.default_rng(n_pts).standard_normal((n, n_pts, 2)).astype(np.float64 if fp64 else np.float32)
            xd = torch.from_numpy(x).cuda()
            a, b = torch.empty_like(xd), torch.empty_like(xd)
            for inv in (0, 1):
                assert run(fp64, n_pts, inv, xd.data_ptr(), a.data_ptr(), b.data_ptr(), n) == 0
                c, s = np.cos(turn), (1 if inv else -1) * np.sin(turn)
                re, im = x[..., 0].astype(wide), x[..., 1].astype(wide)
                ref = np.stack([re @ c - im @ s, re @ s + im @ c], -1)
                err = [float(np.sqrt(((t.cpu().numpy().astype(wide) - ref) ** 2).sum())) for t in (a, b)]
                assert err[0] <= 1.005 * err[1], (n_pts, fp64, inv, err[0] / err[1])


SWEEP_CU = r"""
#include "sweep.cuh"
using namespace ibm;
// lane l: rows of column l, lane-major in f; y, w: [3][ny][32] from half_forward, gl_forward and row by row
template <typename T> __global__ void k(const T *ga, const T *gg, const T *ge, const int *gl, const cplx<T> *f,
                                        cplx<T> *y, T *w, T *q, int *kcs, int ny, int neg) {
  const int l = threadIdx.x, n = gl[l], m = ny;
  const T a = ga[l], g = gg[l], e0 = ge[l];
  const unsigned mask = __ballot_sync(0xffffffffu, n > 0);
  if (n == 0) return;
  cplx<T> *ya = y + l, *yb = ya + 32 * ny, *yc = yb + 32 * ny, e;
  T *wa = w + l, *wb = wa + 32 * ny, *wc = wb + 32 * ny, wk[2], qs[3] = {0, 0, 0};
  for (int s = 0; s < n; ++s) ya[32 * s] = yb[32 * s] = f[32 * s + l];
  half_forward<T>(ya, 32, wa, n, m, a, g, e0, neg != 0, mask, e, qs[0]);
  int kc;
  gl_forward<T, SweepDepth<T>::U>(yb, 32, wb, 32, n, m, a, g, e0, neg != 0, mask, e, qs[1], kc, wk);
  for (int s = kc; s < n; ++s) wb[32 * s] = wk[s & 1];
  T ex = e0, r;
  e = mk<T>(0, 0);
  for (int s = 0; s < n; ++s) {
    ex = sweep_row<T>(a, g, ex, neg != 0, f[32 * s + l], e, qs[2], wc[32 * s], r);
    yc[32 * s] = e;
  }
  for (int v = 0; v < 3; ++v) q[32 * v + l] = qs[v];
  kcs[l] = kc;
}
extern "C" int run(int fp64, const void *a, const void *g, const void *e, const int *len, const void *f, void *y,
                   void *w, void *q, int *kc, int ny, int neg) {
  if (fp64) k<double><<<1, 32>>>((const double *)a, (const double *)g, (const double *)e, len, (const double2 *)f, (double2 *)y, (double *)w, (double *)q, kc, ny, neg);
  else k<float><<<1, 32>>>((const float *)a, (const float *)g, (const float *)e, len, (const float2 *)f, (float2 *)y, (float *)w, (float *)q, kc, ny, neg);
  return (int)cudaDeviceSynchronize();
}
"""


def test_constant_pivots_are_the_recurrences(tmp_path):
    """The half sweeps with their pivots held from the row where the recurrence
    repeats itself, against the recurrence row by row: the same bytes, with
    lanes that differ by a row in length, one that has none, fast and slow
    pencils, both signs and all wall kinds; a good part of the warps goes constant."""
    run = _compiled(tmp_path, "sweep", SWEEP_CU)
    run.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 9 + [ctypes.c_int] * 2
    r = np.random.default_rng(31)
    constant = 0
    for fp64 in (1, 0):
        dt, tdt = (np.float64, torch.float64) if fp64 else (np.float32, torch.float32)
        for trial in range(60):
            ny = int(r.choice([7, 8, 9, 16, 17, 33, 64, 100, 255]))
            ratio = 10.0 ** (r.uniform(-5, 3) + 0.3 * r.random(32))  # g / a, a warp's lanes near one another
            a = np.full(32, 10.0 ** r.uniform(-3, 5))
            g = ratio * a
            e0 = g + a * r.choice([0.0, 1.0, 2.0])
            n = np.where(np.arange(32) % 2 > 0, ny - 1, ny).astype(np.int32)
            n[int(r.integers(32))] = 0
            f = r.standard_normal((ny, 32, 2)).astype(dt)
            args = [dev(v.astype(dt), tdt) for v in (a, g, e0)] + [torch.from_numpy(n).cuda(), torch.from_numpy(f).cuda()]
            y = torch.zeros((3, ny, 32, 2), dtype=tdt, device="cuda")
            w = torch.zeros((3, ny, 32), dtype=tdt, device="cuda")
            q = torch.zeros((3, 32), dtype=tdt, device="cuda")
            kc = torch.zeros(32, dtype=torch.int32, device="cuda")
            out = [y, w, q, kc]
            assert run(fp64, *[t.data_ptr() for t in args + out], ny, int(trial % 2)) == 0
            for v in (0, 1):
                for t in (y, w, q):
                    assert torch.equal(t[v], t[2]), (fp64, ny, v)
            constant += int(kc[n > 0].max()) < ny
    assert constant >= 30

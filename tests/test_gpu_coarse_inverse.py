"""The dense coarsest-level inverses (blocked Gauss-Jordan with partial
pivoting) at the sizes where the blocking can go wrong: fewer nodes than a
panel, whole and ragged panels and update tiles, the largest size, both
operators, several instances of different size in one setup.

Tolerance: the inverse X of A satisfies ||X b - A^-1 b|| <= c N eps cond(A)
||A^-1 b|| with a small c (pivot growth of these stencil matrices is a small
constant); c = 8.  In the complex-FP32 form the stored inverse and the product
are FP32, which adds c eps32 cond(A)."""
import numpy as np
import pytest

import synth
from gpu_util import lib_handle, rnd
from oracle.cycle import CycleParams, Hierarchy, adr_sparse, helmholtz_sparse
from paper_2404_02493_gb300 import binding as B

pytestmark = pytest.mark.gpu


def instance(n, ny, bc="abc1"):
    I = synth.config_layered_rect(n=n, ny=ny, omega=0.4 * (max(n, ny) + 1), bc=bc)
    return I


def check(h, inst, I, ny, n_cmax, prec):
    H = Hierarchy(I.n, I.k, I.phi, I.omega, I.bc, CycleParams(n_cmax=n_cmax, M=1), ny=ny)
    lev = H.lev(H.L)
    N = lev.n * lev.rows
    for which, A in ((0, helmholtz_sparse(lev)), (1, adr_sparse(lev))):
        A = A.toarray()
        dt = np.complex128 if prec == "fp64" else np.complex64
        b = rnd((lev.rows, lev.n), 11 + which, dt)
        x = np.zeros_like(b)
        B.mg_coarse_solve(h, inst, which, b, x)
        ref = np.linalg.solve(A, b.astype(np.complex128).ravel())
        eps = np.finfo(np.float64).eps * N + (np.finfo(np.float32).eps if prec == "mixed" else 0.0)
        err = np.linalg.norm(x.ravel() - ref) / np.linalg.norm(ref)
        assert err <= 8 * eps * np.linalg.cond(A), (which, N, err)


# (n, ny, n_cmax): coarsest 2x2, 3x2, 7x4, 8x8, 15x15, 15x16, 16x16, 31x31, 32x32
SIZES = [(5, 5, 3), (7, 5, 3), (14, 9, 7), (17, 17, 8), (31, 31, 15), (30, 33, 17), (33, 33, 16), (63, 63, 31),
         (65, 65, 32)]


@pytest.mark.parametrize("n,ny,n_cmax", SIZES)
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_coarse_inverse(n, ny, n_cmax, prec):
    I = instance(n, ny)
    p = B.default_params(precision=prec, n_cmax=n_cmax, M=1, autotune=0)
    h = B.mg_setup([(I.n, I.omega, I.k, I.phi, I.bc, ny)], p)
    try:
        if B.mg_num_levels(h) > 2:   # a two-level hierarchy has no ADR operator
            check(h, 0, I, ny, n_cmax, prec)
        else:
            lev_rows = B.mg_level_ny(h, 0, 2), B.mg_level_n(h, 0, 2)
            b = rnd(lev_rows, 3, np.complex128 if prec == "fp64" else np.complex64)
            x = np.zeros_like(b)
            B.mg_coarse_solve(h, 0, 0, b, x)
            H = Hierarchy(I.n, I.k, I.phi, I.omega, I.bc, CycleParams(n_cmax=n_cmax, M=1), ny=ny)
            A = helmholtz_sparse(H.lev(2)).toarray()
            ref = np.linalg.solve(A, b.astype(np.complex128).ravel())
            eps = np.finfo(np.float64).eps * b.size + (np.finfo(np.float32).eps if prec == "mixed" else 0.0)
            assert np.linalg.norm(x.ravel() - ref) <= 8 * eps * np.linalg.cond(A) * np.linalg.norm(ref)
    finally:
        B.mg_destroy(h)


def test_coarse_inverse_batch():
    """Matrices of different size share the launches of one setup."""
    insts = [instance(63, 63), instance(40, 40, "sponge"), instance(127, 127), instance(33, 33, "dirichlet")]
    h = lib_handle(insts, "fp64", n_cmax=15, M=1, autotune=0)
    try:
        for b, I in enumerate(insts):
            check(h, b, I, I.n, 15, "fp64")
    finally:
        B.mg_destroy(h)

"""The planned matvec stages (factor plans of the padded edges, plan_table.h) against
the oracle's FFT matvec: every radix pair class, odd and even edges, columns that are
no multiple of a tile, batches, masks of the mirror groups at thin edges."""
import time

import numpy as np
import pytest
import torch

from oracle import embed, kernel, matvec

vie = pytest.importorskip("paper_1811_00484_gb300")
pytestmark = pytest.mark.gpu

H, F = 5e-3, 298e6
TOL_SVD = 1e-7


def _field(n, B, seed, dtype):
    rng = np.random.default_rng(seed)
    a = rng.standard_normal((B, 3) + n) + 1j * rng.standard_normal((B, 3) + n)
    return torch.from_numpy(a.astype(dtype)).cuda()


def _rel(y, ref):
    y = y.cpu().numpy().astype(np.complex128)
    return np.linalg.norm(y - ref) / np.linalg.norm(ref)


# (n1, n2, n3): every planned edge up to 128 once along some axis, a few beyond, and
# edges without a plan (below 8) beside planned ones
GRIDS = [(8, 9, 10), (12, 14, 15), (16, 18, 20), (21, 24, 25), (27, 28, 30), (32, 7, 35), (36, 40, 4),
         (42, 3, 45), (48, 2, 49), (5, 50, 54), (56, 2, 60), (2, 63, 64), (70, 3, 72), (75, 2, 80),
         (3, 81, 84), (90, 2, 96), (98, 2, 100), (2, 105, 108), (112, 2, 120), (2, 125, 126),
         (128, 2, 12), (9, 2, 128), (135, 2, 8), (2, 8, 140), (2, 150, 9), (8, 2, 160)]


@pytest.mark.parametrize("n", GRIDS)
def test_planned_edges_match_the_oracle(n):
    op = vie.Operator(n, H, F, TOL_SVD, store_uncompressed=True)
    G = embed.green_spectra(kernel.toeplitz_tensor(*n, H, kernel.wavenumber(F)), *n)
    J = _field(n, 3, 7, np.complex64)
    Jh = J.cpu().numpy().astype(np.complex128)
    ref = matvec.matvec_fft(G, Jh)
    adj = matvec.matvec_fft(G, Jh.conj()).conj()              # G is complex symmetric
    # FP32 rounding (1e-5, as for the other FP32 products) plus the truncation 4 tol
    for path, tol in (("tucker", 1e-5 + 4 * TOL_SVD), ("uncompressed", 1e-5)):
        assert _rel(op.matvec(J, path=path), ref) <= tol, path
        assert _rel(op.matvec_adjoint(J, path=path), adj) <= tol, path
    # a row of the batch equals the same current alone, bit for bit
    assert torch.equal(op.matvec(J)[1:2], op.matvec(J[1:2].contiguous()))
    op.close()


@pytest.mark.parametrize("n", [(12, 10, 15), (20, 9, 7)])
def test_ranks_beyond_the_rebuild_kernels(n):
    """A tolerance that keeps every singular vector: the z stage rebuilds in the CTA
    where the rebuild kernels' shared memory does not hold the ranks, and the product
    still meets the FP32 bound."""
    op = vie.Operator(n, H, F, 1e-14)
    G = embed.green_spectra(kernel.toeplitz_tensor(*n, H, kernel.wavenumber(F)), *n)
    J = _field(n, 2, 3, np.complex64)
    assert _rel(op.matvec(J), matvec.matvec_fft(G, J.cpu().numpy().astype(np.complex128))) <= 1e-5
    op.close()


@pytest.mark.parametrize("n", [(8, 8, 8), (7, 9, 10), (16, 12, 24), (5, 24, 18), (20, 21, 15), (3, 14, 16), (10, 24, 24)])
def test_plane_kernel_equals_the_separate_stages(n):
    """Small grids take the y and z stages in one launch; an operator whose rebuild is
    chosen by flag takes them one by one.  Same FP32 rebuild, different radix orders."""
    op, ref = vie.Operator(n, H, F, TOL_SVD, store_uncompressed=True), \
        vie.Operator(n, H, F, TOL_SVD, store_uncompressed=True, rebuild="simt")
    rng = np.random.default_rng(1)
    chi = torch.from_numpy(rng.standard_normal(n) + 1j * rng.standard_normal(n)).cuda()
    for dtype, tol in ((np.complex64, 2e-6), (np.complex128, 2e-14)):   # rounding of two FFT orders
        J = _field(n, 3, 5, dtype)
        c = chi.to(J.dtype)
        for path in ("tucker", "uncompressed"):
            pairs = [(o.matvec(J, path=path), o.apply_system(c, J, path=path),
                      o.apply_system(c, J, adjoint=True, path=path)) for o in (op, ref)]
            for a, b in zip(*pairs):
                assert float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b)) <= tol, (path, dtype)
    # a batch whose right-hand sides converge at different steps
    rhs = torch.cat([_field(n, 1, 8, np.complex64), 0 * _field(n, 1, 8, np.complex64)])
    w, info = op.solve((0.1 * chi).to(torch.complex64), rhs, tol=1e-6)
    w2, info2 = ref.solve((0.1 * chi).to(torch.complex64), rhs, tol=1e-6)
    assert info["converged"] and info2["converged"]
    assert float(torch.linalg.vector_norm(w - w2) / torch.linalg.vector_norm(w2)) <= 1e-4
    op.close()
    ref.close()


def _time(op, J, path="tucker"):
    """Best of eight runs of 20 products, ms."""
    best, (a, b) = float("inf"), (torch.cuda.Event(enable_timing=True) for _ in range(2))
    for _ in range(8):
        op.matvec(J, path=path)
        a.record()
        for _ in range(20):
            op.matvec(J, path=path)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("n", [(32, 8, 32), (16, 24, 24), (20, 20, 20)])
def test_fp64_product_costs_less_than_two(n):
    """The stages spread evenly over the SMs: one right-hand side takes less time than
    two (it took more where CTAs of the next kernel crowded on a few SMs)."""
    op = vie.Operator(n, H, F, 1e-6)
    one, two = (_time(op, _field(n, B, 2, np.complex128)) for B in (1, 2))
    assert one < 0.9 * two, (one, two)
    op.close()


def test_stored_product_costs_no_more_than_the_rebuilt_one():
    """The same in FP32: here the stored path has the same stages and no rebuild."""
    op = vie.Operator((32, 16, 32), H, F, 1e-6, store_uncompressed=True)
    J = _field((32, 16, 32), 8, 2, np.complex64)
    stored, rebuilt = _time(op, J, "uncompressed"), _time(op, J)
    assert stored < rebuilt, (stored, rebuilt)
    op.close()


def test_autotune_times_every_stage_on_plane_grids():
    """The solver runs the separate stages, also where products take the plane kernel:
    the tuner launches each of them for each of its candidates (3 sizes, 4 products)."""
    op = vie.Operator((16, 16, 16), H, F, 1e-6)
    vie.profile_start()
    op.autotune(1)
    ran = vie.profile_stop()
    for f in ("line_x", "line_y", "line_iy", "line_ix"):
        assert ran.get(f, {"launches": 0})["launches"] >= 4 * 3 * 4, (f, ran)
    op.close()


@pytest.mark.parametrize("n", [(12, 10, 7), (12, 30, 45)])
def test_profiler_counts_each_fp64_stage_once(n):
    """x, y, z, inverse y, inverse x, with and without a factor plan for the z edge."""
    op = vie.Operator(n, H, F, 1e-6)
    J = _field(n, 2, 6, np.complex128)
    vie.profile_start(["matvec_fp64"])
    op.matvec(J)
    torch.cuda.synchronize()
    assert vie.profile_stop()["matvec_fp64"]["launches"] == 5
    op.close()


def test_arnoldi_step_of_a_smaller_grid_costs_no_more():
    """One right-hand side, 200 steps in captured cycles: 16^3 and 20^3 against 24^3."""
    best = {}
    for m in (16, 20, 24):
        n = (m, m, m)
        op = vie.Operator(n, H, F, 1e-6)
        g = torch.Generator(device="cuda")
        g.manual_seed(1)
        chi = 5 * torch.randn(n, dtype=torch.complex64, device="cuda", generator=g)
        rhs = torch.randn((1, 3) + n, dtype=torch.complex64, device="cuda", generator=g)
        best[m] = float("inf")
        for _ in range(6):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            _, info = op.solve(chi, rhs, incident=False, tol=1e-13, max_outer=4, refine=False,
                               raise_on_failure=False)
            torch.cuda.synchronize()
            best[m] = min(best[m], time.perf_counter() - t0)
        assert info["iterations"] >= 200
        op.close()
    assert best[16] < 1.1 * best[24] and best[20] < 1.1 * best[24], best

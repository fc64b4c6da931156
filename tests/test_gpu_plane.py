"""The plane kernel (y and z stages of a small grid in one launch) against the oracle, over
the sizes and right-hand sides it is chosen for, in both precisions."""
import numpy as np
import pytest
import torch

from oracle import embed, kernel, matvec

vie = pytest.importorskip("paper_1811_00484_gb300")
pytestmark = pytest.mark.gpu

H, F, TOL = 5e-3, 298e6, 1e-7


def _rel(y, ref):
    y = y.cpu().numpy().astype(np.complex128)
    return np.linalg.norm(y - ref) / np.linalg.norm(ref)


def _launches(f):
    vie.profile_start()
    y = f()
    torch.cuda.synchronize()
    return y, {k: v["launches"] for k, v in vie.profile_stop().items()}


# FP32: each padded edge 16 .. 48 and 56 along y and z, thin and long x; FP64: up to 9 x 9
C64 = [(8, 28, 20), (3, 20, 28), (5, 28, 8), (2, 8, 28), (9, 21, 24), (30, 24, 21), (7, 18, 15), (4, 14, 12),
       (10, 12, 14), (6, 15, 10), (300, 10, 9), (3, 9, 18), (16, 16, 16)]
C128 = [(8, 8, 8), (9, 9, 9), (5, 8, 10), (2, 10, 8), (60, 9, 8)]


@pytest.mark.parametrize("dtype,n", [("c64", n) for n in C64] + [("c128", n) for n in C128])
def test_plane_kernel_matches_the_oracle(dtype, n):
    B = 3 if 2 * n[0] * 3 <= 76 else 1
    op = vie.Operator(n, H, F, TOL, store_uncompressed=True)
    G = embed.green_spectra(kernel.toeplitz_tensor(*n, H, kernel.wavenumber(F)), *n)
    rng = np.random.default_rng(11)
    J = rng.standard_normal((B, 3) + n) + 1j * rng.standard_normal((B, 3) + n)
    J = J.astype(np.complex64 if dtype == "c64" else np.complex128)
    Jd, Jh = torch.from_numpy(J).cuda(), J.astype(np.complex128)
    ref, adj = matvec.matvec_fft(G, Jh), matvec.matvec_fft(G, Jh.conj()).conj()
    eps = 1e-5 if dtype == "c64" else 1e-11            # the other products' bounds
    for path, tol in (("tucker", eps + 4 * TOL), ("uncompressed", eps)):
        y, ran = _launches(lambda: op.matvec(Jd, path=path))
        # x stage, planes, inverse x stage
        if dtype == "c64":
            assert ran["line_x"] == ran["line_ix"] == 1 and "line_y" not in ran, ran
        else:
            assert ran["matvec_fp64"] == 3, ran
        assert _rel(y, ref) <= tol, path
        assert _rel(op.matvec_adjoint(Jd, path=path), adj) <= tol, path
    op.close()


@pytest.mark.parametrize("rebuild", ["mma_sync", "simt", "tcgen05"])
def test_rebuild_kernels_beside_the_planes(rebuild):
    """Rebuild kernels with a ragged H2 = 17 on a grid just outside the plane kernel's
    (P2 P3 = 32 x 96): the kernel that info names is the one that runs."""
    n = (16, 16, 48)
    op = vie.Operator(n, H, F, TOL, rebuild=rebuild)
    assert op.info()["rebuild_kernel"] == rebuild
    G = embed.green_spectra(kernel.toeplitz_tensor(*n, H, kernel.wavenumber(F)), *n)
    rng = np.random.default_rng(12)
    J = (rng.standard_normal((2, 3) + n) + 1j * rng.standard_normal((2, 3) + n)).astype(np.complex64)
    Jd = torch.from_numpy(J).cuda()
    y, ran = _launches(lambda: op.matvec(Jd))
    assert ran["tucker_rebuild"] == 1 and ran["line_y"] == 1, ran
    assert _rel(y, matvec.matvec_fft(G, J.astype(np.complex128))) <= 1e-5 + 4 * TOL
    op.close()

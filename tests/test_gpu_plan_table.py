"""Every factor plan of plan_table.h, as line stage and as z stage, in both precisions, and
the z stage's rebuild inside its CTAs, against the oracle's FFT matvec."""
import os
import re

import numpy as np
import pytest
import torch

from oracle import embed, kernel, matvec

vie = pytest.importorskip("paper_1811_00484_gb300")
pytestmark = pytest.mark.gpu

H, F, TOL = 5e-3, 298e6, 1e-7
TABLE = os.path.join(os.path.dirname(os.path.abspath(vie.__file__)), "csrc", "plan_table.h")
PLANS = sorted(int(m) for m in re.findall(r"^\s+X\((\d+),", open(TABLE).read(), flags=re.M))


def _case(n, B, seed):
    G = embed.green_spectra(kernel.toeplitz_tensor(*n, H, kernel.wavenumber(F)), *n)
    rng = np.random.default_rng(seed)
    J = rng.standard_normal((B, 3) + n) + 1j * rng.standard_normal((B, 3) + n)
    return G, J


def _rel(y, ref):
    y = y.cpu().numpy().astype(np.complex128)
    return np.linalg.norm(y - ref) / np.linalg.norm(ref)


def test_the_table_holds_every_smooth_edge():
    smooth = [N for N in range(16, 513, 2) if not _rest(N)]
    assert PLANS == [N for N in smooth if N != 490]


def _rest(N):
    for p in (2, 3, 5, 7):
        while N % p == 0:
            N //= p
    return N > 1


@pytest.mark.parametrize("N", PLANS)
def test_plan_matches_the_oracle(N):
    """The plan along y (a line stage, three columns) and along z (the z stage; one and two
    mirror lines along x, some groups of a CTA past the last k2)."""
    for n in ((2, N // 2, 3), (3, 2, N // 2)):
        op = vie.Operator(n, H, F, TOL, store_uncompressed=True)
        G, J = _case(n, 2, N)
        for dtype, eps in ((np.complex64, 1e-5), (np.complex128, 1e-11)):   # the products' bounds
            Jd = torch.from_numpy(J.astype(dtype)).cuda()
            Jh = Jd.cpu().numpy().astype(np.complex128)
            ref = matvec.matvec_fft(G, Jh)
            for path, tol in (("uncompressed", eps), ("tucker", eps + 4 * TOL)):
                assert _rel(op.matvec(Jd, path=path), ref) <= tol, (n, path, dtype)
        op.close()


# Ranks so large that the rebuild kernels' shared memory (48 r2 r3 + 384 (r2 + r3) bytes)
# passes 200 KB: P3 = 120 and 128 share a CTA between two groups, 140 has one group per CTA
# (two passes), 270 three passes, 512 the planned 8 x 8 x 8 instead of the kernel that
# needs the scratch; H2 odd, so that the last CTA of a row has a group too many
@pytest.mark.parametrize("n", [(4, 128, 60), (3, 128, 64), (5, 128, 70), (5, 50, 135), (4, 40, 256)])
def test_rebuild_inside_the_z_stage(n):
    op = vie.Operator(n, H, F, 1e-20)                    # every singular vector is kept
    info = op.info()
    assert info["rebuild_kernel"] == "in_cta" and info["rebuild_scratch_bytes"] == 0, info["ranks"]
    G, J = _case(n, 3, 5)
    Jd = torch.from_numpy(J.astype(np.complex64)).cuda()
    Jh = Jd.cpu().numpy().astype(np.complex128)
    assert _rel(op.matvec(Jd), matvec.matvec_fft(G, Jh)) <= 1e-5
    assert _rel(op.matvec_adjoint(Jd), matvec.matvec_fft(G, Jh.conj()).conj()) <= 1e-5
    op.close()

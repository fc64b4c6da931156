"""Setup scratch: components are compressed together only while that costs little memory."""
import math

import numpy as np
import pytest
import torch

vie = pytest.importorskip("paper_1811_00484_gb300")
pytestmark = pytest.mark.gpu

H, F, TOL = 5e-3, 298e6, 1e-6


def _one_component(n, setup):
    """Bytes of the spectrum (spectrum route), one octant, its mode product, the Gram
    matrix and two sets of eigenvectors of every mode, and one factor."""
    h = [m + 1 for m in n]
    entries = 2 * math.prod(h) + 3 * sum(v * v for v in h) + max(h) ** 2
    return 16 * (entries + (8 * math.prod(n) if setup == "spectrum" else 0))


# groups of six, three, two and one component
@pytest.mark.parametrize("n", [(32, 48, 40), (108, 120, 126), (160, 168, 175), (225, 224, 210)])
def test_setup_scratch_is_bounded(n):
    """At most 128 MiB above what one component at a time needs, on both routes, which
    give the same ranks and (4 TOL, both within 2 TOL of the uncompressed one) product."""
    ops = {s: vie.Operator(n, H, F, TOL, setup=s) for s in ("spectrum", "factorwise")}
    for setup, op in ops.items():
        assert op.info()["setup_scratch_bytes"] <= _one_component(n, setup) + 2 ** 27, setup
    a, b = ops.values()
    assert a.info()["ranks"] == b.info()["ranks"]
    for c in range(6):
        for q in range(3):
            sa, sb = a.export(c)[2][q], b.export(c)[2][q]
            r = a.info()["ranks"][c][q]
            # the values above the truncation, whose squares the Gram matrices carry
            assert np.allclose(sa[:r], sb[:r], rtol=1e-6, atol=1e-13 * sa[0])
    g = torch.Generator(device="cuda")
    g.manual_seed(4)
    J = torch.view_as_complex(torch.randn(1, 3, *n, 2, generator=g, device="cuda", dtype=torch.float64))
    y, z = a.matvec(J), b.matvec(J)
    assert float(torch.linalg.vector_norm(y - z) / torch.linalg.vector_norm(y)) <= 4 * TOL
    a.close()
    b.close()

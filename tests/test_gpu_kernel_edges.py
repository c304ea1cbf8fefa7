"""Sizes at which a kernel's tiling or a dispatch rule changes, through the public calls, against the oracle.

The bars are those of the FP64 solver: eigenvalues to 1e-10 relative, principal angles to 1e-8; a product to 1e-12 of each
column's largest entry.
"""
import numpy as np
import pytest

import oracle as O
from paper_1512_06500_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1512_06500_gb300 import build_lib, eda as E
    build_lib.build()
    E.load()
    return E


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


# block widths around the register slices of the Cholesky factorisation with inverse (32, 64, 96 columns) and of one
# warp's rows (8); the wide ones exceed the rank of the problem, so pivots are lost and refilled
@pytest.mark.parametrize("b", [1, 7, 8, 9, 31, 32, 33, 64, 65, 96, 97])
def test_solve_block_width_edges(eda, b):
    p = synth.gaussian_clusters(d=700, k=9, n_per_class=[3, 4, 5, 3, 4, 5, 3, 4, 5], seed=77)
    with eda.build(_dev(p.X), _dev(p.labels), p.k, eda.config(block_b=b, tau=8.0)) as h:
        V, lam, _, info, code = h.solve(p.k - 1, 1e-11)
        assert code == 0, info
        ref = O.eda(p.X, p.labels, p.k, p.k - 1, c2=h.c2, tier="projected")
    V = V.cpu().numpy().T
    assert np.abs(V.T @ V - np.eye(p.k - 1)).max() <= 1e-13
    assert np.max(np.abs(lam.cpu().numpy() - ref["lam_t"]) / ref["lam_t"]) <= 1e-10
    assert O.sin_angle(ref["V"], V) <= 1e-8

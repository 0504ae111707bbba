"""The LLR step's eigen-step on the matrices where it can go wrong: blocks of rank one and two, equal
singular values, all-zero blocks, one to four images, and data at the ends of the float32 range.
Tolerance 1e-5 of the block data, as for the other operators: the threshold weights come from the
float32 Gram matrix, so a component is known to about 6e-8 sigma_max / sigma.  "subnormal" has Gram
matrices below 1e-39, whose 64 products are each rounded to 1.4e-45: 1e-3 of the sum, hence 1e-2."""
import numpy as np
import pytest

import oracle as O

from t2sh_cases import crandn
from test_gpu_parity import OP_TOL, T, c64, host, make_plan, random_problem  # noqa: F401

pytestmark = pytest.mark.gpu


def blocks(rng, kind, K, ny, nz):
    x = crandn(rng, 1, 1, K, ny, nz)
    if kind in ("rank1", "rank2"):
        r = int(kind[-1])
        x = np.einsum("rk,ryz->kyz", crandn(rng, r, K), crandn(rng, r, ny, nz))[None, None]
    elif kind == "equal":   # orthogonal images of equal norm in every block
        x = np.zeros_like(x)
        for k in range(K):
            x[0, 0, k, k % 4::4] = 1.0
    elif kind == "zero":
        x[..., : ny // 2, :] = 0
    elif kind == "tiny":
        x *= 1e-12
    elif kind == "subnormal":
        x *= 1e-21
    elif kind == "huge":
        x *= 1e12
    elif kind == "real":
        x = x.real + 0j
    return x


@pytest.mark.parametrize("kind", ["full", "rank1", "rank2", "equal", "zero", "tiny", "subnormal", "huge", "real"])
@pytest.mark.parametrize("K", [1, 2, 3, 4])
def test_eigen_step(T, kind, K):  # noqa: F811
    rng, phi, mask, maps = random_problem(31 + K, 1, 32, 40, 1, 8, K, 1)
    x = blocks(rng, kind, K, 32, 40).astype(np.complex64)
    scale = float(np.abs(x).max())
    with make_plan(T, phi, mask, maps, block=8) as p:
        for tau in (0.0, 3.0 * scale, 1e3 * scale):
            xg = c64(x)
            p.llr_prox(xg, tau, 0, 4)
            ref = O.llr_prox(x[0].astype(np.complex128), 8, float(np.float32(tau)), 0, 4)
            tol = 1e-2 if kind == "subnormal" else OP_TOL
            assert np.abs(host(xg)[0] - ref).max() <= tol * 8 * scale  # 8: a block's Frobenius norm per entry

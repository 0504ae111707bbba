"""Column and row passes over their whole range of lengths: every size-specialised column and row
length with one and two map sets, enough tiles that a CTA's run crosses column tiles, against the
FP64 oracle.  Tolerance 1e-5: a float32 2D DFT pair accumulates log2(ny nz) <= 18 roundings of
6e-8 per stage, plus the K-term Psi and C-term coil sums, about 1e-6."""
import numpy as np
import pytest

import oracle as O

from t2sh_cases import crandn
from test_gpu_parity import OP_TOL, T, c64, host, make_plan, nrmse, random_problem  # noqa: F401

pytestmark = pytest.mark.gpu

LENGTHS = [
    # S, ny, nz, C, M
    (2, 48, 256, 3, 1),
    (30, 64, 64, 7, 2),      # several column tiles per CTA, short lines
    (3, 96, 192, 2, 1),
    (2, 128, 96, 3, 2),
    (40, 160, 48, 5, 1),     # runs that cross column tiles at 48-point rows
    (1, 192, 160, 2, 2),
    (1, 240, 64, 5, 1),
    (9, 256, 128, 4, 1),
    (5, 260, 240, 6, 1),     # two tensor-map boxes per column
    (20, 260, 64, 12, 1),    # three groups and a spare tile buffer that goes round several times
    (16, 300, 60, 11, 1),    # runs that cross column tiles there
    (21, 234, 52, 7, 2),
    (1, 60, 160, 7, 1),      # coils shared by up to eight CTAs
    (1, 64, 64, 13, 2),
    (3, 78, 240, 6, 2),
    (2, 48, 192, 1, 1),      # one coil
]


@pytest.mark.parametrize("S,ny,nz,C,M", LENGTHS)
def test_passes_of_four_images(T, S, ny, nz, C, M):  # noqa: F811
    rng, phi, mask, maps = random_problem(ny + nz + C, S, ny, nz, C, 12, 4, M)
    x, y = crandn(rng, S, M, 4, ny, nz), crandn(rng, S, C, 4, ny, nz)
    with make_plan(T, phi, mask, maps, block=8) as p:
        got_n, got_a = host(p.normal_op(c64(x))), host(p.adjoint(c64(y), T.KSPACE_PROJ))
        p.sync()
    psi = O.space_time_kernel(mask, phi)
    xs, ys = (a.astype(np.complex64).astype(np.complex128) for a in (x, y))
    for s in {0, S // 2, S - 1}:
        assert nrmse(got_n[s], O.normal(xs[s], maps[s], psi)) < OP_TOL
        assert nrmse(got_a[s], O.adjoint_projected(ys[s], maps[s])) < OP_TOL


@pytest.mark.parametrize("S,ny,nz,C,Tn,K,M", [
    (2, 64, 64, 3, 32, 4, 1),     # exactly one word of echoes
    (1, 256, 48, 5, 33, 4, 2),    # one echo in the second word; planes not a multiple of four
    (3, 260, 160, 3, 70, 4, 1),
    (1, 192, 240, 2, 4, 4, 1),    # as few echoes as images
    (2, 60, 36, 3, 40, 3, 1),     # planar intermediate, K < 4
    (1, 30, 50, 2, 65, 6, 2),     # K > 4
    (1, 16, 24, 1, 7, 4, 1),      # echoes shared out over CTAs: fewer than a chunk,
    (1, 64, 48, 2, 41, 4, 1),     # chunks that end in the second word,
    (3, 256, 160, 8, 40, 4, 1),   # chunks of 32
])
def test_per_echo_and_projected_forms(T, S, ny, nz, C, Tn, K, M):  # noqa: F811
    rng, phi, mask, maps = random_problem(ny + nz + Tn, S, ny, nz, C, Tn, K, M)
    mask[:, ny // 2, nz // 2] = 1   # a point with every echo
    mask[:, 0, :2] = 0              # points with none
    x, y = crandn(rng, S, M, K, ny, nz), crandn(rng, S, C, Tn, ny, nz)
    with make_plan(T, phi, mask, maps) as p:
        te, pr = host(p.forward(c64(x), T.KSPACE_TE)), host(p.forward(c64(x), T.KSPACE_PROJ))
        ad, mu = host(p.adjoint(c64(y), T.KSPACE_TE)), p.step
    xs, ys = (a.astype(np.complex64).astype(np.complex128) for a in (x, y))
    psi = O.space_time_kernel(mask, phi)
    L = max(O.lipschitz(maps[s], psi) for s in range(S))
    assert abs(mu - 1.0 / L) <= 1e-5 / L
    for s in {0, S - 1}:
        ref = O.forward(xs[s], maps[s], mask, phi)
        assert nrmse(te[s], ref) < OP_TOL and np.all(te[s][:, mask == 0] == 0)
        assert nrmse(pr[s], O.project(ref, mask, phi)) < OP_TOL
        assert nrmse(ad[s], O.adjoint(ys[s], maps[s], mask, phi)) < OP_TOL


@pytest.mark.parametrize("S,ny,nz,C,K,M", [
    # every radix of the two-radix passes, chunks of four and of two columns, one to eight images
    (2, 50, 54, 3, 4, 1), (1, 52, 60, 4, 3, 2), (2, 72, 78, 3, 4, 2), (1, 80, 90, 3, 6, 1),
    (3, 100, 104, 2, 2, 1), (1, 108, 120, 5, 4, 1), (1, 130, 144, 2, 5, 2), (2, 150, 156, 2, 4, 1),
    (1, 162, 180, 3, 4, 2), (1, 200, 208, 2, 1, 1), (1, 216, 234, 2, 4, 1), (1, 250, 270, 2, 4, 1),
    (2, 288, 160, 2, 4, 2),   # specialised rows, two-radix columns
    (2, 256, 180, 3, 4, 1),   # specialised columns (rotated slots), two-radix rows
    (1, 128, 100, 3, 4, 2),
    (2, 8, 10, 2, 8, 1), (1, 26, 12, 3, 7, 2),
    (40, 36, 40, 9, 4, 1),    # runs of tiles across column chunks
    (1, 300, 250, 2, 8, 1),   # eight images of 250-point rows: the three-stage passes
    (1, 512, 400, 1, 4, 1),
    (1, 250, 60, 3, 5, 1), (1, 500, 48, 2, 5, 2), (1, 450, 52, 1, 5, 1),  # 25 items of 20 threads: most threads a column CTA has
    # fewer than four images on the planar row lengths, both sides of every line of the choice of layout
    (8, 180, 160, 5, 3, 1), (1, 180, 160, 5, 3, 1), (2, 200, 128, 3, 2, 2), (14, 64, 48, 9, 2, 1), (70, 64, 48, 6, 2, 1),
    (40, 100, 48, 4, 3, 1), (130, 16, 48, 1, 3, 1), (2, 48, 96, 3, 1, 1), (26, 54, 64, 4, 1, 2),
    (1, 64, 338, 2, 4, 1), (1, 90, 512, 2, 2, 1), (1, 390, 16, 2, 2, 1),  # three radix stages: A x in one column pass, and in two
])
def test_two_radix_passes(T, S, ny, nz, C, K, M):  # noqa: F811
    rng, phi, mask, maps = random_problem(ny * nz + K, S, ny, nz, C, 12, K, M)
    x, y = crandn(rng, S, M, K, ny, nz), crandn(rng, S, C, K, ny, nz)
    yt = crandn(rng, S, C, 12, ny, nz)
    with make_plan(T, phi, mask, maps, block=4) as p:
        got_n, got_a = host(p.normal_op(c64(x))), host(p.adjoint(c64(y), T.KSPACE_PROJ))
        got_f, got_t = host(p.forward(c64(x), T.KSPACE_PROJ)), host(p.adjoint(c64(yt), T.KSPACE_TE))
        got_e = host(p.forward(c64(x), T.KSPACE_TE))
    psi = O.space_time_kernel(mask, phi)
    xs, ys, ts = (a.astype(np.complex64).astype(np.complex128) for a in (x, y, yt))
    for s in {0, S // 2, S - 1}:
        ref = O.forward(xs[s], maps[s], mask, phi)
        assert nrmse(got_n[s], O.normal(xs[s], maps[s], psi)) < OP_TOL
        assert nrmse(got_a[s], O.adjoint_projected(ys[s], maps[s])) < OP_TOL
        assert nrmse(got_f[s], O.project(ref, mask, phi)) < OP_TOL
        assert nrmse(got_e[s], ref) < OP_TOL
        assert nrmse(got_t[s], O.adjoint(ts[s], maps[s], mask, phi)) < OP_TOL


COLUMN_LENGTHS = [48, 50, 52, 54, 60, 64, 72, 78, 80, 90, 96, 100, 104, 108, 120, 128, 130, 144, 150, 156, 160, 162,
                  180, 192, 200, 208, 216, 234, 240, 256, 260, 270, 288, 300, 320]


@pytest.mark.parametrize("n", COLUMN_LENGTHS)
def test_every_specialised_length(T, n):  # noqa: F811
    """Four images on every column length, and on every row length that has specialised rows (the
    multiples of four), with one and two map sets, in every direction and form."""
    for ny, nz, M, S, C in [(n, 52, 1, 3, 5), (n, 60, 2, 1, 2)] + ([(54, n, 1, 2, 3), (48, n, 2, 1, 2)] if n % 4 == 0 else []):
        rng, phi, mask, maps = random_problem(ny * nz + M, S, ny, nz, C, 8, 4, M)
        x, y = crandn(rng, S, M, 4, ny, nz), crandn(rng, S, C, 4, ny, nz)
        yt = crandn(rng, S, C, 8, ny, nz)
        with make_plan(T, phi, mask, maps, block=4) as p:
            got_n, got_a = host(p.normal_op(c64(x))), host(p.adjoint(c64(y), T.KSPACE_PROJ))
            got_f, got_t = host(p.forward(c64(x), T.KSPACE_PROJ)), host(p.adjoint(c64(yt), T.KSPACE_TE))
            got_e = host(p.forward(c64(x), T.KSPACE_TE))
        psi = O.space_time_kernel(mask, phi)
        xs, ys, ts = (a.astype(np.complex64).astype(np.complex128) for a in (x, y, yt))
        for s in {0, S - 1}:
            ref = O.forward(xs[s], maps[s], mask, phi)
            assert nrmse(got_n[s], O.normal(xs[s], maps[s], psi)) < OP_TOL
            assert nrmse(got_a[s], O.adjoint_projected(ys[s], maps[s])) < OP_TOL
            assert nrmse(got_f[s], O.project(ref, mask, phi)) < OP_TOL
            assert nrmse(got_e[s], ref) < OP_TOL
            assert nrmse(got_t[s], O.adjoint(ts[s], maps[s], mask, phi)) < OP_TOL


@pytest.mark.parametrize("ny,nz,K", [(64, 48, 4), (50, 54, 4), (36, 30, 6), (96, 64, 2)])
def test_operators_on_odd_views(T, ny, nz, K):  # noqa: F811
    """Arguments that start at an odd value of a larger array (8-byte, not 16-byte aligned) give what
    aligned ones give (per-echo k-space bit for bit; the others may take another pass, so to the
    operators' tolerance), and nothing outside the view is written."""
    import torch

    def odd(shape, v=None):
        n = int(np.prod(shape))
        buf = torch.full((n + 3,), 7.0, dtype=torch.complex64, device="cuda")
        if v is not None:
            buf[1:n + 1] = v.reshape(-1)
        view = buf[1:n + 1].view(shape)
        assert view.data_ptr() % 16 == 8
        return buf, view

    rng, phi, mask, maps = random_problem(ny + nz + K, 2, ny, nz, 3, 11, K, 1)
    x, yt, yp = c64(crandn(rng, 2, 1, K, ny, nz)), c64(crandn(rng, 2, 3, 11, ny, nz)), c64(crandn(rng, 2, 3, K, ny, nz))
    with make_plan(T, phi, mask, maps) as p:
        calls = [(lambda a, o: p.forward(a, T.KSPACE_TE, out=o), x, yt.shape),
                 (lambda a, o: p.forward(a, T.KSPACE_PROJ, out=o), x, yp.shape),
                 (lambda a, o: p.adjoint(a, T.KSPACE_TE, out=o), yt, x.shape),
                 (lambda a, o: p.adjoint(a, T.KSPACE_PROJ, out=o), yp, x.shape),
                 (lambda a, o: p.normal_op(a, out=o), x, x.shape)]
        for call, a, shape in calls:
            ref = call(a, torch.empty(shape, dtype=torch.complex64, device="cuda"))
            buf, out = odd(shape)
            call(odd(a.shape, a)[1], out)
            torch.cuda.synchronize()
            assert torch.equal(out, ref) if shape == yt.shape else nrmse(host(out), host(ref)) < OP_TOL
            assert buf[0] == 7 and bool((buf[-2:] == 7).all())
        p.sync()


def test_chained_operators_see_the_previous_result(T):  # noqa: F811
    """Every kernel may start while the one before it still runs: operators chained on one array give the
    bits that they give with a synchronisation after each, over many repetitions."""
    import torch

    rng, phi, mask, maps = random_problem(7, 6, 54, 50, 5, 20, 4, 1)   # rows that share DRAM sectors
    x0 = c64(crandn(rng, 6, 1, 4, 54, 50))
    with make_plan(T, phi, mask, maps) as p:
        def chain(sync):
            x, y = x0.clone(), torch.empty((6, 5, 20, 54, 50), dtype=torch.complex64, device="cuda")
            for i in range(8):
                p.forward(x, T.KSPACE_TE, out=y), sync()
                p.adjoint(y, T.KSPACE_TE, out=x), sync()
                p.llr_prox(x, 0.01, i % 4, i % 3), sync()
                p.normal_op(x, out=x), sync()
            torch.cuda.synchronize()
            return x
        ref = chain(torch.cuda.synchronize)
        assert bool(torch.isfinite(torch.view_as_real(ref)).all()) and float(ref.abs().max()) > 0
        for _ in range(20):
            assert torch.equal(chain(lambda: None), ref)
        p.sync()

"""GPU checks of the fp32-precision tensor-core paths at the sizes where their tilings can go wrong: long lists
(kernels of their own), tile remainders, ranks around the tile widths, the factorisation's blocks."""
import math

import numpy as np
import pytest
import torch

from oracle import fira_oracle as fo
from paper_2410_01623_b200 import binding as fb
from paper_2410_01623_b200 import workloads as wk
from tests.parity_util import Trajectory, residual_jump, to_np64

pytestmark = pytest.mark.gpu

# remainders of every extent, both orientations, ranks that are no multiple of 4 or 8, above one tile (128) and above
# the width up to which accumulators are double-buffered (256)
BASE = [(150, 333), (333, 150), (130, 130), (64, 200), (257, 129), (129, 257), (300, 1000), (1000, 300), (512, 700), (7, 9),
        (640, 512), (512, 256)]
RANKS = [36, 37, 64, 16, 100, 128, 200, 255, 130, 3, 300, 128]


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("flags,ranks", [(0, RANKS), (0, [r // 4 * 4 or 4 for r in RANKS]), (fb.FLAG_MATRIX_SCALING, RANKS),
                                         (fb.FLAG_NO_RESIDUAL, RANKS), (fb.FLAG_ONLY_SCALING, RANKS),
                                         (fb.FLAG_PSI_RMSPROP, RANKS), (fb.FLAG_PSI_ADAGRAD, RANKS)])
def test_long_list_of_ragged_matrices(dtype, flags, ranks):
    """A list of many elements takes kernels of its own in fp32 precision (step variants, row lengths that are and are not
    multiples of four).  From moments of ordinary size: on a first step N = R / (|R| + eps) is the sign of R, and among
    some 10^6 entries of R a few lie within fp32's error of zero, where that sign, and with it a column of the update, is
    not determined."""
    g = torch.Generator().manual_seed(11)
    hp = fb.make_hparams(lr=1e-2, alpha=0.25, gamma=1.01, flags=flags | fb.FLAG_FORCE_SIMT)
    W0 = [(torch.randn(m, n, generator=g) * 0.02).to(dtype) for m, n in BASE * 4]
    tr = Trajectory(BASE * 4, ranks * 4, dtype, hp, W0)
    Ps = []
    for i, (m, n) in enumerate(tr.shapes):
        q, _ = torch.linalg.qr(torch.randn(min(m, n), tr.f.ranks[i], generator=g, dtype=torch.float64))
        Ps.append(q.to(dtype))
        tr.f.set_projection(i, Ps[i].cuda())
        V = torch.rand(max(m, n), tr.f.ranks[i], generator=g) + 0.5
        tr.f.set_state(i, torch.zeros_like(V).cuda(), V.cuda(), 1e6, 3)
        tr.st[i].V, tr.st[i].prev_norm, tr.st[i].t = to_np64(V.T if m <= n else V).copy(), 1e6, 3
    for step in range(3):
        G = [torch.randn(m, n, generator=g).to(dtype) for m, n in tr.shapes]
        tr.step([residual_jump(x, p) for x, p in zip(G, Ps)] if step == 2 else G)
    tr.assert_ok()
    assert all(tr.f.diagnostics(i)["engine"] == 0 for i in range(len(BASE)))
    assert flags & fb.FLAG_NO_RESIDUAL or any(l < 1.0 for l in tr.lams[-1])
    assert tr.f.last_step_launches() > 4


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_long_list_with_pitches_and_in_chunks(dtype):
    """The same list with padded rows, whole and as the host path's chunks: the same weights as without padding, bit for
    bit (the order of every sum is the same), and the padding untouched."""
    shapes, ranks = BASE * 4, [r // 4 * 4 or 4 for r in RANKS] * 4
    g = torch.Generator().manual_seed(5)
    hp = fb.make_hparams(lr=1e-2, alpha=0.25, gamma=1.01, flags=fb.FLAG_FORCE_SIMT)
    lds = [n + (3, 8, 0)[i % 3] for i, (m, n) in enumerate(shapes)]
    fs = [fb.Fira(shapes, ranks, dtype, hp), fb.Fira(shapes, ranks, dtype, hp, lds=lds), fb.Fira(shapes, ranks, dtype, hp)]
    W0 = [(torch.randn(m, n, generator=g) * 0.02).to(dtype) for m, n in shapes]
    for i, (m, n) in enumerate(shapes):
        P = torch.linalg.qr(torch.randn(min(m, n), ranks[i], generator=g, dtype=torch.float64))[0].to(dtype).cuda()
        for f in fs:
            f.set_projection(i, P)
    Wa = [w.cuda() for w in W0]
    Wb = [torch.full((m, ld), 7.0, dtype=dtype, device="cuda") for (m, n), ld in zip(shapes, lds)]
    Gb = [torch.full((m, ld), float("nan"), dtype=dtype, device="cuda") for (m, n), ld in zip(shapes, lds)]
    for w, b, (m, n) in zip(W0, Wb, shapes):
        b[:, :n] = w.cuda()
    Wh = [w.clone().pin_memory() for w in W0]
    staging = torch.empty(fs[2].staging_bytes(), dtype=torch.uint8, device="cuda")
    for _ in range(2):
        G = [torch.randn(m, n, generator=g).to(dtype) for m, n in shapes]
        for x, b, (m, n) in zip(G, Gb, shapes):
            b[:, :n] = x.cuda()
        fs[0].step(Wa, [x.cuda() for x in G])
        fs[1].step(Wb, Gb)
        fs[2].step_host(Wh, [x.pin_memory() for x in G], staging)
        torch.cuda.synchronize()
    assert [f.poll() for f in fs] == [0, 0, 0]
    for i, (m, n) in enumerate(shapes):
        assert torch.equal(Wa[i], Wb[i][:, :n]), (i, shapes[i])
        assert torch.equal(Wa[i].cpu(), Wh[i]), (i, shapes[i])
        assert (Wb[i][:, n:] == 7.0).all()


@pytest.mark.parametrize("shape,r", [((300, 420), 1), ((300, 420), 127), ((420, 300), 128), ((300, 420), 129),
                                     ((700, 515), 257), ((384, 1024), 384)])
def test_refresh_at_the_edges_of_its_blocks(shape, r):
    """Bases whose Gram factor has one row, one block less one, whole blocks, one row in its last block, and full rank:
    orthonormal to fp32 and the SVD's subspace."""
    m, n = shape
    G = wk.planted_gradient(m, n, r, seed=r, gap=4.0).cuda() if r < min(m, n) else torch.randn(m, n, generator=torch.Generator().manual_seed(3)).cuda()
    f = fb.Fira([shape], r, torch.float32, fb.make_hparams())
    f.refresh_projection([G], seed=12, iters=6)
    assert f.poll() == 0
    P = to_np64(f.get_projection(0))
    assert np.abs(P.T @ P - np.eye(r)).max() < 1e-5
    if r < min(m, n):
        assert fo.principal_angles(P, fo.refresh_projection(to_np64(G), r)).max() <= 1e-3


def _stepped_from_ordinary_moments(shapes, ranks, dtype, flags, steps=3, seed=11):
    """See test_long_list_of_ragged_matrices; the last step's gradient jumps."""
    g = torch.Generator().manual_seed(seed)
    hp = fb.make_hparams(lr=1e-2, alpha=0.25, gamma=1.01, flags=flags | fb.FLAG_FORCE_SIMT)
    tr = Trajectory(shapes, ranks, dtype, hp, [(torch.randn(m, n, generator=g) * 0.02).to(dtype) for m, n in shapes])
    Ps = []
    for i, (m, n) in enumerate(shapes):
        q, _ = torch.linalg.qr(torch.randn(min(m, n), ranks[i], generator=g, dtype=torch.float64))
        Ps.append(q.to(dtype))
        tr.f.set_projection(i, Ps[i].cuda())
        V = torch.rand(max(m, n), ranks[i], generator=g) + 0.5
        tr.f.set_state(i, torch.zeros_like(V).cuda(), V.cuda(), 1e6, 3)
        tr.st[i].V, tr.st[i].prev_norm, tr.st[i].t = to_np64(V.T if m <= n else V).copy(), 1e6, 3
    for step in range(steps):
        G = [torch.randn(m, n, generator=g).to(dtype) for m, n in shapes]
        tr.step([residual_jump(x, p) for x, p in zip(G, Ps)] if step == steps - 1 else G)
    return tr


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("flags", [0, fb.FLAG_MATRIX_SCALING, fb.FLAG_NO_SCALING, fb.FLAG_ONLY_SCALING])
@pytest.mark.parametrize("shapes,ranks", [([(333, 517), (517, 333)], [129, 200]), ([(640, 900), (900, 640)], [300, 640]),
                                          ([(1100, 1376)], [1000])])
def test_short_list_of_ranks_above_one_tile(shapes, ranks, flags, dtype):
    """Row sums over several tiles of R, factors made from them, products longer than one piece of the main accumulator;
    grids of fewer and of more tiles than SMs, and a list that a rank above 512 keeps short."""
    tr = _stepped_from_ordinary_moments(shapes, ranks, dtype, flags)
    tr.assert_ok()
    assert all(tr.f.diagnostics(i)["engine"] == 0 for i in range(len(shapes)))


def test_more_tiles_than_sms_with_ranks_above_one_tile():
    _stepped_from_ordinary_moments([(512, 1376)] * 4, [200] * 4, torch.float32, 0, steps=2).assert_ok()


def test_projection_split_over_blocks_of_more_than_one_piece():
    """44 tiles of R: two blocks per tile, 256 of k each."""
    _stepped_from_ordinary_moments([(512, 1376), (1376, 512)] * 2, [128] * 4, torch.float32, 0).assert_ok()


@pytest.mark.parametrize("shapes,r", [([(520, 1376)], 200), ([(520, 1376)], 512), ([(1100, 1376)], 1024),
                                      ([(520, 1376), (1376, 520)] * 5, 256), ([(520, 1376), (1376, 520)] * 5, 512)])
def test_long_products_do_not_drift(shapes, r):
    """Products of positive numbers, W = -lr alpha Pi N alone.  An MMA adds to its accumulator by truncation, which loses half
    a unit in the last place on average: 0.72 / 2 2^-23 = 4.3e-8 of the running sum.  Over the 8 additions of one piece
    of 128 that is 4.5 / 8 of it each, 1.9e-7 in all, and the pieces are added to nearest; the whole of k in one
    accumulator gives 3.7e-7 at 256 and twice that at 512.  A bound of 2e-7 lies between."""
    f = fb.Fira(shapes, r, torch.float32, fb.make_hparams(lr=1.0, alpha=1.0, beta1=0.0, beta2=0.5, flags=fb.FLAG_NO_RESIDUAL))
    g = torch.Generator(device="cuda").manual_seed(5)
    W, G, P = [], [], []
    for i, (m, n) in enumerate(shapes):
        P.append(torch.randn(min(m, n), r, generator=g, device="cuda").abs())
        G.append(torch.randn(m, n, generator=g, device="cuda").abs())
        W.append(torch.zeros(m, n, device="cuda"))
        V = torch.rand(max(m, n), r, generator=g, device="cuda") + 0.5
        f.set_projection(i, P[i])
        f.set_state(i, torch.zeros_like(V), V, None, 100)
    f.step(W, G)
    for i, (m, n) in enumerate(shapes):
        M, V, _, _ = f.get_state(i)
        N = (1 - 0.5 ** 101) ** 0.5 * M.double() / (V.double().sqrt() + 1e-8)
        D = P[i].double() @ N.T if m <= n else N @ P[i].double().T
        assert abs(float((-W[i].double() - D).sum() / D.sum())) < 2e-7


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("flags", [0, fb.FLAG_MATRIX_SCALING, fb.FLAG_NO_RESIDUAL, fb.FLAG_PSI_RMSPROP])
@pytest.mark.parametrize("shapes,ranks", [([(130, 65), (65, 130), (64, 129), (129, 63), (200, 192)], [33, 32, 31, 5, 128]),
                                          ([(512, 1376)], [128]), ([(384, 1030)] * 3, [100] * 3)])
def test_short_list_that_steps_in_one_kernel(shapes, ranks, flags, dtype):
    """Half tiles of W and their edges, ranks around the slabs' depth, a rank of whole slabs; whole tiles (81 of them)."""
    tr = _stepped_from_ordinary_moments(shapes, ranks, dtype, flags)
    tr.assert_ok()
    assert tr.f.last_step_launches() == 2


@pytest.mark.parametrize("shapes,ranks,launches", [([(1100, 2800), (512, 1376), (1376, 512)], [64, 200, 128], 4),
                                                   ([(1200, 3840), (512, 1376)], [100, 128], 7)])
def test_long_list_around_the_tiles_of_one_kernel(shapes, ranks, launches):
    """fp32 matrices of more tiles than CTA pairs, whose pairs have two tiles of one matrix, and of more than twice as many, which
    take two kernels."""
    tr = _stepped_from_ordinary_moments(shapes, ranks, torch.float32, 0)
    tr.assert_ok()
    assert tr.f.last_step_launches() == launches


@pytest.mark.parametrize("shapes,ranks", [(wk.llama_shapes(8, 288, 992), [64] * 56), (wk.llama_shapes(20, 160, 416), [40] * 140),
                                          ([(1024, 32)] * 80 + [(1024, 1024)] * 5, [16] * 80 + [128] * 5)])
def test_long_list_with_runs_of_narrow_tiles(shapes, ranks):
    """Tiles whose last columns number 32 or fewer have one box of W where others have four: of the loader's buffers five such tiles
    take no more than one wide one.  Pairs with four and more of them in a row and a wide tile, or one of another rank, behind."""
    tr = _stepped_from_ordinary_moments(shapes, ranks, torch.float32, 0)
    tr.assert_ok()
    assert tr.f.last_step_launches() == 4
    g = torch.Generator().manual_seed(3)
    fs = [fb.Fira(shapes, ranks, torch.float32, fb.make_hparams(lr=1e-2, alpha=0.25, gamma=1.01)) for _ in range(2)]
    for i, (m, n) in enumerate(shapes):
        P = torch.linalg.qr(torch.randn(min(m, n), ranks[i], generator=g))[0].contiguous().cuda()
        for f in fs:
            f.set_projection(i, P)
    Wh = [(torch.randn(s, generator=g) * 0.02).pin_memory() for s in shapes]
    W = [w.cuda() for w in Wh]
    staging = torch.empty(fs[1].staging_bytes(), dtype=torch.uint8, device="cuda")
    for _ in range(2):
        G = [torch.randn(s, generator=g).pin_memory() for s in shapes]
        fs[0].step(W, [x.cuda() for x in G])
        fs[1].step_host(Wh, G, staging)
        torch.cuda.synchronize()
    assert [f.poll() for f in fs] == [0, 0]
    assert all(torch.equal(w.cpu(), h) for w, h in zip(W, Wh))


def _squares(total, count):
    """`count` whole numbers of at most 90 whose squares add up to total."""
    out = np.zeros(count)
    whole, rest = divmod(total, 8100)
    out[:whole] = 90
    four = next((a, b, c, e) for a in range(91) for b in range(a + 1) for c in range(b + 1)
                for e in [math.isqrt(max(0, rest - a * a - b * b - c * c))] if a * a + b * b + c * c + e * e == rest)
    out[whole:whole + 4] = four
    return out


@pytest.mark.parametrize("dtype,launches", [(torch.float32, 4), (torch.bfloat16, 7)])
def test_norm_of_long_lists_loses_nothing_between_tiles(dtype, launches):
    """||S|| of whole numbers.  What one warp adds up in fp32 is exact (2048 squares of 90 at most: below 2^24).  A tile's sum takes 28 bits
    and lies 7 above a multiple of 16, which rounding it to 24 bits takes off in each of 32 tiles; the whole lies 2 to 18
    above the square of the middle between two fp32 numbers.  So the norm is the upper one only if nothing is rounded in between."""
    shapes = [(1024, 1024)] * 6
    f = fb.Fira(shapes, 64, dtype, fb.make_hparams(flags=fb.FLAG_NO_SCALING | fb.FLAG_FORCE_SIMT))      # P = 0: S = G
    Gs, want = [], []
    for i in range(len(shapes)):
        low = np.float32(92000 + 17 * i)
        middle = (float(low) + float(np.spacing(low)) / 2) ** 2
        total = (int(middle) // 16 + 1) * 16
        total += 16 * (total - middle < 2)
        G = np.zeros((1024, 1024))
        sums = [total // 32 // 16 * 16 + 7] * 32
        sums[-1] += total - sum(sums)
        for t, x in enumerate(sums):
            assert x % 16 == 7 and 2 ** 27 < x < 2 ** 28
            G[t // 8 * 256:t // 8 * 256 + 256, t % 8 * 128:t % 8 * 128 + 128] = _squares(x, 256 * 128).reshape(256, 128)
        assert (G * G).sum() == total
        Gs.append(torch.from_numpy(G).to(dtype).cuda())
        want.append(float(np.nextafter(low, np.float32(np.inf))))
        assert want[-1] == float(np.float32(math.sqrt(total)))
    f.step([torch.zeros(1024, 1024, dtype=dtype, device="cuda") for _ in shapes], Gs)
    assert f.poll() == 0 and f.last_step_launches() == launches
    assert [f.diagnostics(i)["norm_scaled"] for i in range(len(shapes))] == want


@pytest.mark.parametrize("shapes,flags,names", [
    ([(512, 1376)], 0, ["k_project", "k_back_step"]),
    ([(512, 1376)] * 8, 0, ["k_project", "k_moments", "k_part_step"]),
    ([(512, 1376)], fb.FLAG_ONLY_SCALING, ["k_project", "k_moments", "k_back_project<norm>", "k_finalize", "k_form_x", "k_back_project<update>"])])
def test_phase_times_name_the_kernels_that_ran(shapes, flags, names):
    f = fb.Fira(shapes, 128, torch.float32, fb.make_hparams(flags=flags))
    W, G = ([torch.randn(s, device="cuda") for s in shapes] for _ in range(2))
    f.refresh_projection(G)
    f.step(W, G)
    f.enable_phase_timing()
    for _ in range(3):
        f.step(W, G)
    phases, steps = f.phase_times()
    assert [k for k, _ in phases] == names and steps == 3
    assert flags or all(ms > 1e-3 for _, ms in phases)

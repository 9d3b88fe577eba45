"""The 2D FP32 strips (one warp per 28 columns) and the FP32 and double-word batches built on them,
against the oracle at the sizes where a strip can go wrong: meshes narrower than
a strip, its edges and remainders, chunks of rows and their remainders, every
boundary rule, groups of 1D strips; and one mesh of more than 2^30 cells (64-bit
offsets)."""
import numpy as np
import pytest

import oracle as O
from paper_1207_3392_gb300 import hydro as H
from paper_1207_3392_gb300 import problems as P
from parity_util import TOL_FP32, TOL_FP64, check, oracle_run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1207_3392_gb300 import build
    build.build()
    yield


@pytest.mark.parametrize("bc", [P.PERIODIC, P.REFLECT, P.OUTFLOW])
@pytest.mark.parametrize("n", [(2, 2), (3, 9), (27, 5), (28, 33), (29, 4), (56, 3), (57, 38), (226, 7)])
def test_strip_edges_match_the_oracle(n, bc):
    pr = P.random_blocks(2, n, seed=40 + n[0], bc=bc).with_(grad_phi=(0.2, -0.3, 0.0))
    for solver in (H.HLL, H.HLLC):
        Uo, to = oracle_run(pr, solver=solver, steps=3)
        ref = None
        for tile in (0, 1, 2):
            for kc in (0, 1, 4, 5):
                h = H.Hydro.from_problem(pr, precision=H.FP32_MIXED, solver=solver)
                h.set_tile(tile, kc)
                t = h.advance(3, pr.cfl)
                U = h.get_conserved(precision=H.FP64)
                tot = h.step_totals()
                h.close()
                assert t == pytest.approx(to, rel=1e-5)
                if ref is None:
                    ref, ref_tot = U, tot
                    check(U, Uo, 2, TOL_FP32, f"{n} bc={bc} solver={solver}")
                np.testing.assert_array_equal(U, ref, err_msg=f"tile {tile} kchunk {kc}")
                # the same cells summed in another grouping: 48-bit sums
                np.testing.assert_allclose(tot, ref_tot, rtol=1e-12, atol=1e-12 * np.max(np.abs(ref_tot)))


@pytest.mark.parametrize("precision,tol", [(H.FP32_MIXED, TOL_FP32), (H.FP64_DW, TOL_FP64)])
def test_batch_of_edge_sizes_matches_the_oracle(precision, tol):
    probs = [P.random_blocks(1, (m,), seed=m, bc=bc) for m in (2, 27, 28, 29, 223, 224, 225, 449)
             for bc in (P.PERIODIC, P.REFLECT, P.OUTFLOW)]
    probs += [P.random_blocks(2, m, seed=m[0], bc=P.REFLECT) for m in ((2, 2), (28, 31), (29, 33), (57, 65))]
    b = H.Batch(probs, precision=precision)
    for i, pr in enumerate(probs):
        b.set_primitive(i, pr.rho, pr.vel, pr.p)
    b.run(4, 0.4)
    assert b.status() == -1
    for i, pr in enumerate(probs):
        Uo, _ = oracle_run(pr.with_(cfl=0.4), steps=4)
        check(b.get_conserved(i), Uo, pr.ndim, tol, f"problem {i} {pr.n}")
    b.close()


def test_mesh_beyond_2_30_cells():
    """A Sod tube along x on 65536 x 16400 cells: sampled rows, up to the last,
    are bitwise the first row and match the 1D oracle step."""
    import torch
    nx, ny = 65536, 16400
    if torch.cuda.mem_get_info()[0] < 90e9:
        pytest.skip("needs 90 GB of device memory")
    pr = P.sod(nx)
    g = O.Grid(pr)
    U1 = O.initial_state(pr, g).astype(np.float32)
    U = torch.zeros((4, ny, nx), dtype=torch.float32, device="cuda")
    for v, a in zip((0, 1, 3), U1):
        U[v] = torch.from_numpy(a).cuda()
    h = H.Hydro(2, (nx, ny), [pr.widths[0], np.full(ny, 1.0)], (P.OUTFLOW,) * 2, (P.OUTFLOW,) * 2, 1.4, H.HLLC,
                precision=H.FP32_MIXED)
    torch.cuda.synchronize()
    h.set_conserved(U)
    dt = h.compute_dt(0.4)
    h.step(dt)
    h.get_conserved(U)
    h.close()
    rows = U[:, [0, 1, ny // 2, ny - 2, ny - 1]].cpu().numpy()
    del U
    torch.cuda.empty_cache()
    for k in range(1, rows.shape[1]):
        np.testing.assert_array_equal(rows[:, k], rows[:, 0])
    Uo = O.step(g, U1.astype(np.float64), dt)
    check(rows[[0, 1, 3], 0].astype(np.float64), Uo, 1, TOL_FP32, "wide mesh")


@pytest.mark.parametrize("precision,tol,tile", [(H.FP32_MIXED, TOL_FP32, 14), (H.FP64_DW, TOL_FP64, 4)])
@pytest.mark.parametrize("bc", [P.PERIODIC, P.REFLECT, P.OUTFLOW])
@pytest.mark.parametrize("n", [(2, 2, 2), (3, 5, 3), (27, 4, 5), (28, 7, 4), (29, 3, 9), (57, 9, 11), (226, 3, 14)])
def test_split_stages_match_the_oracle_and_the_tiles(n, bc, precision, tol, tile):
    """3D on independent warps (a launch for x and y, one for z): planes of 4 k
    cells (the shared-memory ring) and of other counts, chunks of planes and
    their remainders; bitwise the state of tile 0."""
    pr = P.random_blocks(3, n, seed=60 + n[0], bc=bc).with_(grad_phi=(0.2, -0.3, 0.1))
    for solver in (H.HLL, H.HLLC):
        Uo, to = oracle_run(pr, solver=solver, steps=2)
        ref = None
        for t, kc in ((tile, 0), (tile, 1), (tile, 3), (tile, 8), (0, 0)):
            h = H.Hydro.from_problem(pr, precision=precision, solver=solver)
            h.set_tile(t, kc)
            time = h.advance(2, pr.cfl)
            U = h.get_conserved(precision=H.FP64)
            tot = h.step_totals()
            h.close()
            if ref is None:
                ref, ref_tot = U, tot
                assert time == pytest.approx(to, rel=1e-5 if tol == TOL_FP32 else 1e-10)
                check(U, Uo, 3, tol, f"{n} bc={bc} solver={solver}")
            np.testing.assert_array_equal(U, ref, err_msg=f"tile {t} kchunk {kc}")
            np.testing.assert_allclose(tot, ref_tot, rtol=1e-12, atol=1e-12 * np.max(np.abs(ref_tot)))


@pytest.mark.parametrize("n", [(2, 2), (27, 5), (29, 33), (57, 38)])
def test_double_word_strips_match_the_oracle_and_the_tiles(n):
    for bc in (P.PERIODIC, P.REFLECT, P.OUTFLOW):
        pr = P.random_blocks(2, n, seed=80 + n[0], bc=bc)
        Uo, _ = oracle_run(pr, steps=3)
        ref = None
        for t, kc in ((1, 0), (1, 1), (1, 5), (0, 0)):
            h = H.Hydro.from_problem(pr, precision=H.FP64_DW)
            h.set_tile(t, kc)
            h.advance(3, pr.cfl)
            U = h.get_conserved()
            h.close()
            if ref is None:
                ref = U
                check(U, Uo, 2, TOL_FP64, f"dw {n} bc={bc}")
            np.testing.assert_array_equal(U, ref, err_msg=f"tile {t} kchunk {kc}")


@pytest.mark.parametrize("n", [(36, 5, 4), (20, 10, 8), (2, 34, 5), (3, 12, 4)])
def test_split_cfl_speed_on_a_mesh_refined_towards_the_upper_walls(n):
    """Planes of 4 k cells that are not whole warps of the z march, the smallest
    cells at the upper end of x (of y where a row is shorter than 4 cells) and the
    fastest sound just before them: dt is the largest cell speed's, and dt, time
    and state are those of tile 0 bit for bit."""
    pr = P.random_blocks(3, n, seed=5, bc=P.REFLECT)
    axis = 0 if n[0] >= 4 else 1
    widths = [np.full(m, 0.01) for m in n]
    widths[axis] *= 0.6 ** np.maximum(0, np.arange(n[axis]) - (n[axis] - 5))
    p = np.ones(pr.shape)
    if axis == 0:
        p[:, n[1] - 1, n[0] - 4:n[0] - 1] = 9.0
    else:
        p[:, n[1] - 2, :] = 9.0
    pr = pr.with_(widths=widths, rho=np.ones(pr.shape), vel=np.zeros_like(pr.vel), p=p)
    cs = np.sqrt(pr.gamma * p)
    iw = [1.0 / w.reshape([-1 if a == 2 - q else 1 for a in range(3)]) for q, w in enumerate(widths)]
    dt = 0.3 / max(np.max(cs * i) for i in iw)
    ref = None
    for tile, kc in ((14, 0), (14, 1), (14, 3), (0, 0)):
        h = H.Hydro.from_problem(pr, precision=H.FP32_MIXED)
        h.set_tile(tile, kc)
        first = h.advance(1, 0.3)
        assert first == pytest.approx(dt, rel=1e-6), f"tile {tile} kchunk {kc}"
        out = first, h.advance(3, 0.3), h.get_conserved()
        h.close()
        ref = ref or out
        assert out[:2] == ref[:2], f"tile {tile} kchunk {kc}"
        np.testing.assert_array_equal(out[2], ref[2])


@pytest.mark.parametrize("precision,tile", [(H.FP32_MIXED, {2: 0, 3: 14}), (H.FP64_DW, {2: 1, 3: 4})])
@pytest.mark.parametrize("n", [(30, 9, 7), (57, 33)])
def test_totals_in_any_unit_of_length_and_density(n, precision, tile):
    """Widths times 2^66 (areas beyond FP32's range), widths times 2^-40 and
    densities and pressures times 2^-30 (shares below 2^-102): the totals scale by
    exactly that power of two, and without a scale they are FP64's to 2^-45."""
    pr = P.random_blocks(len(n), n, seed=7)
    got = {}
    for lw, ls in ((0, 0), (66, 0), (-40, 0), (-20, -30)):
        h = H.Hydro.from_problem(pr.with_(widths=[w * 2.0 ** lw for w in pr.widths], rho=pr.rho * 2.0 ** ls,
                                          p=pr.p * 2.0 ** ls), precision=precision)
        h.set_tile(tile[len(n)], 0)
        U0 = h.get_conserved(precision=H.FP64)
        h.advance(1, 0.3)
        got[lw, ls] = np.array(h.step_totals()) / 2.0 ** (len(n) * lw + ls)
        h.close()
        if lw == ls == 0:
            vol = np.ones(pr.shape)
            for q in range(len(n)):
                vol = vol * np.asarray(pr.widths[q]).reshape([-1 if a == len(n) - 1 - q else 1 for a in range(len(n))])
            ref = np.array([np.sum(u * vol) for u in U0])
            size = np.array([np.sum(np.abs(u) * vol) for u in U0])
            assert np.all(np.abs(got[0, 0] - ref) <= 2.0 ** -45 * size)
        np.testing.assert_array_equal(got[lw, ls], got[0, 0], err_msg=f"widths 2^{lw}, state 2^{ls}")


@pytest.mark.parametrize("precision,n,tile", [(H.FP32_MIXED, (2, 65535 * 32 + 1), 0), (H.FP64_DW, (2, 65535 * 32 + 1), 1),
                                              (H.FP32_MIXED, (2, 2, 65535 * 48 + 1), 14)])
def test_march_axis_beyond_65535_chunks(precision, n, tile):
    """A march axis of more chunks than a grid has along z, at the automatic chunk
    and at a requested one of one row: bitwise the state of long chunks."""
    nd = len(n)
    rng = np.random.default_rng(3)
    shape = tuple(reversed(n))
    rho, p = rng.uniform(0.5, 2.0, shape), rng.uniform(0.5, 2.0, shape)
    vel = rng.uniform(-0.5, 0.5, (nd,) + shape)
    ref = None
    for kc in (64, 0, 1):
        h = H.Hydro(nd, n, [np.full(m, 0.1) for m in n], (P.OUTFLOW,) * nd, (P.REFLECT,) * nd, 1.4, H.HLLC,
                    precision=precision)
        assert kc or h.tile_info()["tile"] == tile
        h.set_tile(tile, kc)
        h.set_primitive(rho, vel, p)
        h.advance(1, 0.4)
        U = h.get_conserved()
        h.close()
        ref = U if ref is None else ref
        np.testing.assert_array_equal(U, ref, err_msg=f"kchunk {kc}")


@pytest.mark.parametrize("precision", [H.FP32_MIXED, H.FP64_DW])
def test_batch_results_do_not_depend_on_the_strips_per_item(precision):
    """1D problems at the edges of strips and of groups of strips, alone (one strip
    an item), beside 1D meshes that make the items 2 to 8 strips, and beside a 2D
    one (8): the same bits."""
    probs = [P.random_blocks(1, (m,), seed=m, bc=bc) for m in (2, 28, 29, 56, 57, 85, 113, 141, 197, 224, 225, 449)
             for bc in (P.PERIODIC, P.OUTFLOW)]
    ref = None
    for cells in (0, 200000, 500000, 1500000, -1):
        more = [P.random_blocks(1, (cells,), seed=1, bc=P.REFLECT)] if cells > 0 else []
        if cells < 0:
            more = [P.random_blocks(2, (60, 40), seed=1, bc=P.REFLECT)]
        b = H.Batch(probs + more, precision=precision)
        for i, pr in enumerate(probs + more):
            b.set_primitive(i, pr.rho, pr.vel, pr.p)
        b.run(4, 0.4)
        assert b.status() == -1
        got = [b.get_conserved(i) for i in range(len(probs))]
        if more:
            h = H.Hydro.from_problem(more[0], precision=precision)
            h.advance(4, 0.4)
            np.testing.assert_array_equal(b.get_conserved(len(probs)), h.get_conserved(precision=H.FP64))
            h.close()
        b.close()
        ref = ref or got
        for a, c in zip(got, ref):
            np.testing.assert_array_equal(a, c, err_msg=f"{cells} cells beside")


@pytest.mark.parametrize("precision,n,tile", [(H.FP32_MIXED, (29, 40, 40), 14), (H.FP32_MIXED, (32, 128, 160), 14),
                                              (H.FP32_MIXED, (32, 128, 161), 0), (H.FP32_MIXED, (33, 160, 160), 14),
                                              (H.FP64_DW, (32, 64, 128), 4), (H.FP64_DW, (32, 64, 129), 0)])
def test_default_tile_of_3d_meshes_one_tile_wide(precision, n, tile):
    pr = P.random_blocks(3, n, seed=3)
    for solver in (H.HLLC, H.HLLC_SWITCH)[:2 if precision == H.FP32_MIXED else 1]:
        h = H.Hydro.from_problem(pr, precision=precision, solver=solver)
        assert h.tile_info()["tile"] == tile
        h.advance(1, 0.3)
        U = h.get_conserved()
        h.set_primitive(pr.rho, pr.vel, pr.p)
        h.set_tile(14 - tile if precision == H.FP32_MIXED else 4 - tile, 0)
        h.advance(1, 0.3)
        np.testing.assert_array_equal(h.get_conserved(), U)
        h.close()

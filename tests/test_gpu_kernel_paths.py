"""GPU: which kernel and tile serve a grid under GABP_KERNEL_AUTO, against the split kernels (the
plain form of the iteration), bit for bit, at the sizes where the choice changes."""
import numpy as np
import pytest

import gabp_synth
from gpu_common import decode_messages, ensure_built, solver, sorted_obs_order

pytestmark = pytest.mark.gpu

SPLIT = 2


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def _problem(nx, ny, seed=5):
    return gabp_synth.make_problem(nx, ny, 0.05, seed, n_tracks=4, per_track=max(nx, ny), n_uniform=max(nx * ny // 15, 2),
                                   sigma=(0.02, 0.1))


@pytest.mark.parametrize("shape, tile", [((2, 2), (8, 4)), ((8, 4), (8, 4)), ((9, 5), (8, 4)), ((64, 3), (8, 4)),
                                         ((63, 61), (8, 4)), ((120, 120), (8, 4)), ((120, 121), (16, 4)),
                                         ((256, 152), (16, 4)), ((257, 153), (16, 8)), ((256, 300), (16, 8)),
                                         ((273, 421), (16, 14))])
def test_fp64_auto_tiles_match_split(shape, tile):
    p = _problem(*shape)
    bufs = []
    for kernel in (SPLIT, 0):
        with solver(p, "fp64", kernel=kernel) as s:
            if kernel == 0:
                st = s.stats()
                assert (st["tile_x"], st["tile_y"]) == tile
            s.iterate(23, 0.3)
            bufs.append(s.get_messages())
    assert np.array_equal(bufs[0], bufs[1])


@pytest.mark.parametrize("shape", [(45, 38), (145, 138)])
def test_fp64_interior_update_with_a_prior_mean_matches_split(shape):
    p = _problem(*shape)
    fb = np.random.default_rng(1).standard_normal(p.n)
    bufs = []
    for kernel in (SPLIT, 0):
        with solver(p, "fp64", kernel=kernel) as s:
            s.set_prior_mean(fb)
            s.iterate(15, 0.5)
            bufs.append(s.get_messages())
    assert np.array_equal(bufs[0], bufs[1])


@pytest.mark.parametrize("gamma", [3e-303, 1e-150, 1e150, 1e303])
def test_fp64_reciprocals_out_of_the_fast_range(orc, gamma):
    """Scales whose precisions leave 2^+-1000 take the divisions: the marginals are the oracle's."""
    p = gabp_synth.make_problem(20, 18, 0.3, 2, n_uniform=60)
    fl = orc.build_factors(p.nx, p.ny, p.kappa, p.obs_x, p.obs_y, p.y, p.noise_var, gamma)
    with np.errstate(all="ignore"):
        mu_o, var_o, _ = orc.gabp(fl, 0.5, 12)
    with solver(p, "fp64", gamma=gamma) as s:
        s.iterate(12, 0.5)
        mu, var = s.marginals()
    ok = np.isfinite(mu_o) & np.isfinite(var_o)
    np.testing.assert_allclose(mu[ok], mu_o[ok], rtol=1e-10, atol=1e-10 * np.max(np.abs(mu_o[ok])))
    np.testing.assert_allclose(var[ok], var_o[ok], rtol=1e-10)


@pytest.mark.parametrize("shape", [(5, 820), (61, 68), (62, 67), (63, 66), (90, 46), (91, 46), (1021, 7), (331, 209)])
def test_fp32_padded_rows_match_split(shape):
    """Widths that are not a multiple of 4, from 4096 nodes on: the TMA kernel on padded plane rows.
    Messages, checkpoints (whose layout has no padding), message change, warm start, residual and
    marginals are those of the split kernels."""
    p = _problem(*shape)
    got = []
    for kernel in (SPLIT, 0):
        with solver(p, "fp32", kernel=kernel) as s:
            assert s.stats()["kernel"] == (SPLIT if kernel else 3)
            s.iterate(23, 0.3)
            a = s.get_messages()
            change, res = s.message_change(), s.residual()
            s.iterate(4, 0.3)
            s.set_messages(a)
            s.iterate(4, 0.3)
            b = s.get_messages()
            mean, var = s.marginals()
            s.warm_start(mean, 1.0 / var)
            s.iterate(3, 0.3)
            got.append((a, b, s.get_messages(), mean, var, np.array([change, res])))
    for x, y in zip(*got):
        # the message change adds the planes in another order of threads (the padded layout)
        np.testing.assert_allclose(x, y, rtol=1e-5) if x.size == 2 else np.testing.assert_array_equal(x, y)


def test_fp32_small_or_tiled_odd_grids_keep_the_sweep():
    for (nx, ny), opts in [((63, 65), {}), ((91, 70), dict(tile_x=30, tile_y=32)), ((4, 2), {})]:
        p = _problem(nx, ny)
        with solver(p, "fp32", **opts) as s:
            assert s.stats()["kernel"] == (3 if nx == 4 else 4)
    from paper_2404_12968_gb300 import GabpError
    with pytest.raises(GabpError, match="multiple of 4"):
        solver(_problem(91, 70), "fp32", kernel=3)   # asked for by name: as before


@pytest.mark.parametrize("shape, per_cell, tile", [((4, 2), 9, 2), ((32, 32), 25, 2), ((60, 59), 3, 2), ((90, 100), 1, 2), ((90, 101), 1, 6),
                                                   ((91, 102), 5, 6), ((130, 67), 2, 6), ((301, 160), 3, 6),
                                                   ((300, 300), 1, 14)])
def test_fp32_short_tiles_match_split(shape, per_cell, tile):
    """The short TMA tiles of small and of densely observed grids (tiles shared by several blocks, the
    belief sums of many observations per node) against the split kernels."""
    nx, ny = shape
    rng = np.random.default_rng(11)
    m = per_cell * nx * ny + 1
    # half of the observations on one corner cell of every fourth column: long, uneven ranges
    xy = rng.uniform(0, 1, (m, 2)) * np.array([nx - 1.0, ny - 1.0])
    xy[::2, 0] = np.minimum(np.floor(xy[::2, 0] / 4) * 4, nx - 2) + 0.5
    y, nv = rng.standard_normal(m), rng.uniform(0.01, 0.1, m)
    from paper_2404_12968_gb300 import Solver
    bufs = []
    for kernel in (SPLIT, 0):
        with Solver(nx=nx, ny=ny, kappa=0.2, obs_xy=xy, y=y, noise_var=nv, precision="fp32", kernel=kernel) as s:
            if kernel == 0 and nx % 4 == 0 or nx * ny >= 4096:
                assert kernel or (s.stats()["kernel"], s.stats()["tile_y"]) == (3, tile)
            s.iterate(23, 0.5)
            bufs.append(s.get_messages())
    assert np.array_equal(bufs[0], bufs[1])


@pytest.mark.gpu
@pytest.mark.parametrize("B,H,W", [(1, 8, 8), (2, 40, 72), (3, 24, 136)])
def test_network_gradients_on_ragged_tiles(B, H, W):
    """Weight and bias gradients of the tensor-core kernels (16 x 8 pixel tiles, the bias summed from
    the same tiles) against the mma.sync kernels and their separate bias kernel: both are within 6 % of
    the reference in BF16 (test_gpu_warmstart.py), so within 12 % of each other; a lost or doubled tile
    of these grids is a larger share."""
    torch = pytest.importorskip("torch")
    from oracle import unet
    from paper_2404_12968_gb300 import (GABP_WSNET_MMA_SYNC, GABP_WSNET_TCGEN05, WarmStartNet,
                                        gabp_wsnet_gradients, gabp_wsnet_set_kernels)
    net = WarmStartNet(seed=11, device=0)
    rng = np.random.default_rng(12)
    offs, head, total = unet.layout()
    net.set_params((net.params() + rng.normal(size=total) * 0.02).astype(np.float32))
    x = torch.zeros((B, H, W, 16))
    x[..., :3] = torch.tensor(rng.normal(size=(B, H, W, 3)))
    x = x.to(torch.bfloat16).view(torch.int16).cuda()
    t = torch.tensor(rng.normal(size=(B, H, W, 2)) + 2.0, dtype=torch.float32).cuda()
    grads = []
    for k in (GABP_WSNET_TCGEN05, GABP_WSNET_MMA_SYNC):
        gabp_wsnet_set_kernels(net.handle, k)
        g = np.empty(total, np.float32)
        gabp_wsnet_gradients(net.handle, list(x), list(t), H, W, g)
        grads.append(g)
    net.close()
    for i, (wo, bo) in enumerate(offs):
        for lo, hi in [(wo, bo), (bo, bo + unet.SPECS[i][1])]:
            a, b = grads[0][lo:hi], grads[1][lo:hi]
            assert np.linalg.norm(a - b) < 0.12 * np.linalg.norm(b), (i, lo)


@pytest.mark.parametrize("shape, per_node", [((23, 89), 3), ((64, 32), 3), ((683, 3), 6), ((31, 199), 2), ((128, 160), 0.02)])
def test_observation_index_at_block_edges(orc, shape, per_node):
    """The observation index is formed 2048 cells at a time: node counts around multiples of 2048,
    many observations per cell and few; |b| and the residual gather over it."""
    nx, ny = shape
    p = gabp_synth.make_problem(nx, ny, 0.3, 9, n_uniform=int(per_node * nx * ny), sigma=(0.05, 0.2))
    fl = orc.build_factors(nx, ny, p.kappa, p.obs_x, p.obs_y, p.y, p.noise_var)
    mu_o, var_o, _ = orc.gabp(fl, 0.5, 6)
    with solver(p, "fp64") as s:
        s.iterate(6, 0.5)
        mu, var = s.marginals()
        assert s.residual() == pytest.approx(orc.residual(fl, mu), rel=1e-8)
    np.testing.assert_allclose(mu, mu_o, rtol=1e-10, atol=1e-10 * np.max(np.abs(mu_o)))
    np.testing.assert_allclose(var, var_o, rtol=1e-10)


def test_batch_residuals_of_very_uneven_members():
    """One grid of 352 blocks among grids of one: the batch's residual kernels give a member four times
    the average member's blocks (68), so the large one strides.  The same sums as a single context."""
    from paper_2404_12968_gb300 import Batch
    probs = [_problem(300, 300)] + [_problem(8 + i, 8, seed=i) for i in range(20)] + [gabp_synth.make_problem(9, 8, 0.1, 4)]
    with Batch(probs, tile_y=14) as b:
        for iters in (8, 7):   # both message buffers
            b.iterate(iters, 0.3)
            res = b.residuals()
        for i, p in enumerate(probs):
            with solver(p, "fp32") as s:
                s.iterate(15, 0.3)
                assert s.residual() == res[i], i


@pytest.mark.parametrize("m", [1, 31, 33, 1024, 1025, 4097, 16383, 16384, 16385])
@pytest.mark.parametrize("shape", [(2, 3), (19, 13), (201, 330)])
def test_observation_sort_in_one_block(orc, m, shape):
    """Up to 16384 observations one block sorts them, beyond that the passes over many: the stable
    order by base cell, for cell counts of one, two and three 8-bit digits, with many ties."""
    nx, ny = shape
    rng = np.random.default_rng(m + nx)
    x, y = rng.uniform(0, nx - 1, m), rng.uniform(0, ny - 1, m)
    x[m // 3:m // 2], y[m // 3:m // 2] = 0.5, ny - 1.0
    p = gabp_synth.Problem(nx, ny, 0.3, x, y, rng.normal(size=m), rng.uniform(0.01, 0.2, m))
    order, base, w = sorted_obs_order(orc, p)
    with solver(p, "fp64") as s:
        _, obs = decode_messages(s.get_messages(), p, "fp64")
    np.testing.assert_allclose(obs[:, :, 1], (w ** 2 / p.noise_var[:, None])[order], rtol=1e-12, atol=0)

"""The 2D FP64 sweep at the edges of its blocks against the oracle: extents around the 16-column moment
blocks and below them, odd rows in the last band, bands of one and of many rows, velocity counts that fill a
16-velocity group, leave one nearly empty, and need one row per warp (more than 256 per quadrant)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle
from paper_1712_01132_gb300 import dvm, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1,n2,nv,rows,tile,opts", [
    (3, 3, 4, 0, 0, {}), (15, 7, 6, 0, 0, {}), (16, 5, 8, 1, 8, {}), (17, 9, 8, 3, 16, {}),
    (33, 31, 8, 32, 8, {}), (31, 40, 10, 5, 8, {"lateral": "specular"}), (50, 21, 18, 0, 0, {}),
    (19, 6, 34, 0, 0, {}), (35, 7, 34, 2, 8, {"specular_fraction": 0.3}), (18, 5, 44, 0, 16, {}),
    (40, 33, 12, 7, 0, {"specular_fraction": 0.6, "lateral": "specular"}),
    (37, 29, 8, 0, 0, {"subdomains": (3, 2, 1)}), (36, 12, 34, 3, 0, {"subdomains": (2, 3, 1)}),
    (20, 18, 8, 0, 0, {"stencil_order": 1})])
def test_matches_oracle(n1, n2, nv, rows, tile, opts):
    rng = np.random.default_rng(n1 * 100 + n2)
    mask = rng.random((n2, n1)) < 0.3
    mask[n2 // 2, n1 // 2], mask[0, 0] = True, False
    opts = dict({"lateral": "periodic"}, **opts)
    v, w = dvm.dvm_gh_velocity_grid(2, nv)
    s = dvm.Solver(mask, 0.2, v, w, precision="fp64", band_rows=rows, tile_x1=tile, **opts)
    o = oracle.Oracle(mask, 0.2, v, w, lateral=opts["lateral"], order=opts.get("stencil_order", 2),
                      alpha=1.0 - opts.get("specular_fraction", 0.0), decomposition=opts.get("subdomains", (1, 1)))
    for n in (1, 2, 9):
        s.step(n)
        s.sync()
        o.iterate(n)
        (rho, u), (rho_o, u_o) = s.moments(), o.moments()
        # FP64 sums of at most 1936 velocities over 12 iterations, in another order: 1e-12 of the largest value
        assert np.abs(u - u_o).max() < 1e-12 * max(1.0, np.abs(u_o).max())
        assert np.abs(rho - rho_o).max() < 1e-12 * max(1.0, np.abs(rho_o).max())


@pytest.mark.parametrize("n1", [33, 49, 97])
@pytest.mark.parametrize("nv", [10, 16, 24])
def test_velocity_groups_share_their_sums(n1, nv):
    """Two and more velocity groups a unit and three and more blocks of 16 columns: the groups' sums of a block and of the
    one after next go through the same buffer.  Two runs give the same bits, and the oracle's moments."""
    mask = np.random.default_rng(n1 + nv).random((11, n1)) < 0.3
    mask[5, n1 // 2], mask[0, 0] = True, False
    v, w = dvm.dvm_gh_velocity_grid(2, nv)
    runs = []
    for _ in range(2):
        s = dvm.Solver(mask, 0.2, v, w, precision="fp64", lateral="periodic")
        s.step(12)
        s.sync()
        runs.append(s.moments())
    o = oracle.Oracle(mask, 0.2, v, w, lateral="periodic")
    o.iterate(12)
    for got, again, want in zip(runs[0], runs[1], o.moments()):
        assert np.array_equal(got, again)
        assert np.abs(got - want).max() < 1e-12 * max(1.0, np.abs(want).max())      # as above


@pytest.mark.parametrize("opts", [{}, {"specular_fraction": 0.4}])
def test_expired_wait_inside_a_band_is_reported(opts):
    """One band, for which no other waits: records that never come make the waits between its warps expire (64 x 1 ms).
    The call reports DVM_ETIMEOUT, whichever warp gave up, and the context iterates normally afterwards."""
    mask = np.zeros((9, 40), bool)
    mask[4, 7:20] = True
    v, w = dvm.dvm_gh_velocity_grid(2, 8)
    s = dvm.Solver(mask, 0.2, v, w, precision="fp64", lateral="periodic", band_rows=16, **opts)
    s.debug_set_wait(1_000_000, withhold_item=-2)
    s.step(1)
    with pytest.raises(dvm.DvmError) as ei:
        s.sync()
    assert ei.value.status == dvm.DVM_ETIMEOUT
    s.debug_set_wait(2_000_000_000)
    s.step(3)
    s.sync()
    assert np.isfinite(s.moments()[1]).all()


@pytest.mark.parametrize("n1,n2,nv,tile", [(200, 45, 8, 8), (131, 30, 16, 8), (90, 11, 34, 16)])
def test_edges_through_a_short_ring(n1, n2, nv, tile):
    """Many bands, whose edges pass through rings far shorter than a row (one lane waits for the band below, all lanes
    copy): two runs give the same bits, and the oracle's moments."""
    mask = np.random.default_rng(n1).random((n2, n1)) < 0.25
    mask[n2 // 2, n1 // 2], mask[0, 0] = True, False
    v, w = dvm.dvm_gh_velocity_grid(2, nv)
    runs = []
    for _ in range(2):
        s = dvm.Solver(mask, 0.2, v, w, precision="fp64", lateral="periodic", tile_x1=tile)
        s.step(8)
        s.sync()
        runs.append(s.moments())
    o = oracle.Oracle(mask, 0.2, v, w, lateral="periodic")
    o.iterate(8)
    for got, again, want in zip(runs[0], runs[1], o.moments()):
        assert np.array_equal(got, again)
        assert np.abs(got - want).max() < 1e-12 * max(1.0, np.abs(want).max())      # as above


@pytest.mark.parametrize("n1,n2,nv,rows,opts", [
    (37, 9, 16, 8, {}), (35, 11, 22, 4, {}), (50, 5, 32, 0, {}), (33, 4, 44, 0, {}), (34, 9, 8, 32, {}),
    (35, 6, 32, 0, {"specular_fraction": 0.5}), (36, 8, 22, 4, {"subdomains": (2, 2, 1)})])
def test_sixteen_sweeping_warps(n1, n2, nv, rows, opts):
    """Bands of 16 sweeping warps, which have moment warps (and a register bound) of their own."""
    mask = np.random.default_rng(n1 + n2).random((n2, n1)) < 0.3
    mask[n2 // 2, n1 // 2], mask[0, 0] = True, False
    v, w = dvm.dvm_gh_velocity_grid(2, nv)
    s = dvm.Solver(mask, 0.2, v, w, precision="fp64", lateral="periodic", band_rows=rows, **opts)
    o = oracle.Oracle(mask, 0.2, v, w, lateral="periodic", alpha=1.0 - opts.get("specular_fraction", 0.0),
                      decomposition=opts.get("subdomains", (1, 1)))
    s.step(10)
    s.sync()
    o.iterate(10)
    for got, want in zip(s.moments(), o.moments()):
        assert np.abs(got - want).max() < 1e-12 * max(1.0, np.abs(want).max())      # as above

"""The tile kernel at the sizes where its bond draws and its row labelling
change course: rows that start on an odd site (odd L: a row's draws reach into
a 65th Philox block), tiles of at most 64 columns (half the blocks drawn), tile
widths around each 32-site word and tile heights around each sub-tile row.
Integers, so every comparison with the oracle is exact."""
import numpy as np
import pytest

from gpu_util import assert_obs_equal

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sw():
    import __graft_entry__
    __graft_entry__.build()
    from paper_0808_2109_gb300 import swgpu
    swgpu.lib()
    return swgpu


@pytest.mark.parametrize("tile_h", [32, 64, 96, 128])
@pytest.mark.parametrize("L", [61, 66, 126, 161, 191, 193, 223, 225, 259])
def test_word_and_subtile_edges(sw, orc, L, tile_h):
    for T, opts in ((2.0, {}), (2.269185, {"csize": True, "open": True}), (3.0, {})):
        ref = orc.sw_chain(L, 1.0, T, L, **opts)
        with sw.Lattice(L, T=T, seed=L, tile_h=tile_h, **opts) as lat:
            for n in (1, 3):   # the first sweep of a call reads its spins from memory
                lat.sweep(n)
                assert_obs_equal(lat.observables(), ref.run(n))
                np.testing.assert_array_equal(lat.spins(), ref.spin)
                np.testing.assert_array_equal(lat.labels(), ref.label)
                np.testing.assert_array_equal(lat.bonds(), ref.bond)


# Potts tiles (128 x 64, 32 x 16 x 16): word edges and odd rows in 2D; in 3D
# row blocks of 4 x 8, quarter words at their boundaries, and rows that start
# at every place of a Philox block.  With and without csize (labels then keep
# their roots' indices) and with the table's last states (q = 256).
@pytest.mark.parametrize("csize", [False, True])
@pytest.mark.parametrize("dim,L,q", [(2, 63, 3), (2, 66, 2), (2, 126, 256), (2, 191, 3), (2, 193, 2),
                                     (3, 5, 2), (3, 12, 256), (3, 15, 3), (3, 18, 2), (3, 31, 2), (3, 47, 3),
                                     (3, 52, 2)])
def test_potts_word_and_block_edges(sw, orc, dim, L, q, csize):
    tc = 1.0 / np.log(1 + np.sqrt(q)) if dim == 2 else (2.2557 if q == 2 else 1.8164)
    for T in (0.8 * tc, tc, 1.5 * tc):
        ref = orc.PottsChain(dim, L, q, 1.0, T, L, csize=csize)
        with sw.PottsLattice(dim, L, q, T=T, seed=L, csize=csize) as lat:
            for n in (1, 3):
                lat.sweep(n)
                assert_obs_equal(lat.observables(), ref.run(n))
                np.testing.assert_array_equal(lat.spins(), ref.spin)
                np.testing.assert_array_equal(lat.labels(), ref.label)
                np.testing.assert_array_equal(lat.bonds(), ref.bond)


# Lattices of a single tile run all sweeps of a call in one block.
@pytest.mark.parametrize("opts", [{}, {"open": True}])
@pytest.mark.parametrize("L,tile_h", [(2, 0), (3, 128), (31, 0), (32, 32), (33, 0), (63, 96), (64, 0), (65, 0),
                                      (96, 96), (97, 0), (127, 0), (128, 0)])
def test_one_tile_lattices(sw, orc, L, tile_h, opts):
    for T in (1.5, 2.269185, 3.5):
        ref = orc.sw_chain(L, 1.0, T, L, **opts)
        with sw.Lattice(L, T=T, seed=L, tile_h=tile_h, **opts) as lat:
            for n in (1, 4):
                lat.sweep(n)
                assert_obs_equal(lat.observables(), ref.run(n))
                np.testing.assert_array_equal(lat.spins(), ref.spin)
                np.testing.assert_array_equal(lat.labels(), ref.label)
                np.testing.assert_array_equal(lat.bonds(), ref.bond)


def test_one_tile_call_longer_than_a_launch(sw, orc):
    ref = orc.sw_chain(12, 1.0, 2.269185, 5)
    with sw.Lattice(12, T=2.269185, seed=5) as lat:
        lat.sweep(4099)   # a launch runs at most 4096 sweeps
        assert_obs_equal(lat.observables(), ref.run(4099))
        np.testing.assert_array_equal(lat.spins(), ref.spin)
        np.testing.assert_array_equal(lat.labels(), ref.label)


@pytest.mark.parametrize("L", [2, 33, 96, 128])
def test_static_sweep_of_one_tile(sw, L):
    torch = pytest.importorskip("torch")
    thr = sw.sw_threshold(1.0, 2.269185)
    with sw.Lattice(L, p=thr / 2.0 ** 32, seed=7) as ref:
        spins = torch.from_numpy(ref.spins()).cuda()
        out, labels = torch.empty_like(spins), torch.empty(L * L, dtype=torch.int32, device="cuda")
        obs = torch.full((sw.OBS_DTYPE.itemsize,), 0xAB, dtype=torch.uint8, device="cuda")
        for k in range(2):
            sw.sw_sweep_static((spins if k == 0 else out).data_ptr(), out.data_ptr(), labels.data_ptr(),
                               obs.data_ptr(), L, thr, 7, k, torch.cuda.current_stream())
            torch.cuda.synchronize()
            ref.sweep(1)
            assert obs.cpu().numpy().tobytes() == ref.observables().tobytes()
            np.testing.assert_array_equal(out.cpu().numpy(), ref.spins())
            np.testing.assert_array_equal(labels.cpu().numpy(), ref.labels())


# The height that a lattice gets without asking, at both sides of the rule's lines.
@pytest.mark.parametrize("L,opts", [(64, {"csize": True}), (65, {"csize": True}), (65, {"pcc": True}),
                                    (128, {"wind": True}), (129, {}), (384, {"wind": True}), (385, {"wind": True}),
                                    (512, {"pcc": True}), (513, {"pcc": True}), (1920, {}), (1921, {}),
                                    (30, {"wind": True}), (768, {"wind": True}), (769, {"wind": True}),
                                    (1056, {"wind": True, "csize": True}), (1057, {"wind": True, "csize": True}),
                                    (1536, {"pcc": True}), (1537, {"pcc": True})])
def test_default_heights(sw, orc, L, opts):
    kw = {"pcc": True} if "pcc" in opts else {"T": 2.269185}
    rest = {k: v for k, v in opts.items() if k != "pcc"}
    with sw.Lattice(L, seed=L, **kw, **rest) as lat, sw.Lattice(L, seed=L, tile_h=64, **kw, **rest) as ref:
        for n in (1, 3):
            lat.sweep(n)
            ref.sweep(n)
            assert lat.observables().tobytes() == ref.observables().tobytes()
            np.testing.assert_array_equal(lat.spins(), ref.spins())
            np.testing.assert_array_equal(lat.labels(), ref.labels())
            np.testing.assert_array_equal(lat.bonds(), ref.bonds())


@pytest.mark.parametrize("L", [129, 512, 513, 1024])   # 32-row tiles up to L = 512
def test_static_sweep_of_tiles(sw, L):
    torch = pytest.importorskip("torch")
    thr = sw.sw_threshold(1.0, 2.269185)
    with sw.Lattice(L, p=thr / 2.0 ** 32, seed=7, tile_h=96) as ref:
        spins = torch.from_numpy(ref.spins()).cuda()
        out, labels = torch.empty_like(spins), torch.empty(L * L, dtype=torch.int32, device="cuda")
        obs = torch.empty(sw.OBS_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
        sw.sw_sweep_static(spins.data_ptr(), out.data_ptr(), labels.data_ptr(), obs.data_ptr(), L, thr, 7, 0,
                           torch.cuda.current_stream())
        torch.cuda.synchronize()
        ref.sweep(1)
        assert obs.cpu().numpy().tobytes() == ref.observables().tobytes()
        np.testing.assert_array_equal(out.cpu().numpy(), ref.spins())
        np.testing.assert_array_equal(labels.cpu().numpy(), ref.labels())


# 32-row tiles have sub-tiles of 8, 16 or 32 rows by the size of the grid.
@pytest.mark.parametrize("opts", [{}, {"csize": True, "open": True}, {"pcc": True}, {"wind": True}])
@pytest.mark.parametrize("L", [609, 801, 846, 1939, 1985])
def test_rows_of_subtiles(sw, L, opts):
    kw = {"pcc": True} if "pcc" in opts else {"T": 2.269185}
    rest = {k: v for k, v in opts.items() if k != "pcc"}
    with sw.Lattice(L, seed=L, tile_h=32, **kw, **rest) as lat, sw.Lattice(L, seed=L, tile_h=96, **kw, **rest) as ref:
        for n in (1, 3):
            lat.sweep(n)
            ref.sweep(n)
            assert lat.observables().tobytes() == ref.observables().tobytes()
            np.testing.assert_array_equal(lat.spins(), ref.spins())
            np.testing.assert_array_equal(lat.labels(), ref.labels())
            np.testing.assert_array_equal(lat.bonds(), ref.bonds())


# Potts tiles have 32, 16 or 8 warps by the size of the grid (the sizes above: 32).
@pytest.mark.parametrize("opts", [{}, {"csize": True, "open": True}, {"wind": True}])
@pytest.mark.parametrize("dim,L,q", [(2, 1290, 3), (2, 1681, 2), (3, 97, 3), (3, 161, 2)])
def test_potts_warps_of_a_tile(sw, orc, dim, L, q, opts):
    T = 1.0 / np.log(1 + np.sqrt(q)) if dim == 2 else (2.2557 if q == 2 else 1.8164)
    ref = orc.PottsChain(dim, L, q, 1.0, T, L, **opts)
    with sw.PottsLattice(dim, L, q, T=T, seed=L, **opts) as lat:
        for n in (1, 2):
            lat.sweep(n)
            assert_obs_equal(lat.observables(), ref.run(n))
            np.testing.assert_array_equal(lat.spins(), ref.spin)
            np.testing.assert_array_equal(lat.labels(), ref.label)
            np.testing.assert_array_equal(lat.bonds(), ref.bond)


@pytest.mark.parametrize("dim,L", [(2, 200), (2, 1290), (3, 40), (3, 97)])
def test_potts_pcc_warps_of_a_tile(sw, orc, dim, L):
    ref = orc.PottsChain(dim, L, 2, 1.0, 1.0, 3, pcc=True)
    with sw.PottsLattice(dim, L, 2, seed=3, pcc=True) as lat:
        lat.sweep(4)
        assert_obs_equal(lat.observables(), ref.run(4))
        np.testing.assert_array_equal(lat.spins(), ref.spin)

"""Every shape of the tile kernels against the oracle under every option: 32-row
tiles with sub-tiles of 8, 16 and 32 rows, default heights at the lines of their
rule, Potts tiles of 32, 16 and 8 warps with PCC.  Integers, exact."""
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


def _check(lat, ref, opts):
    """A call of one sweep and one of two; a PCC chain then once more from ordered
    spins, where (at the threshold of the hot start) some cluster spans."""
    spans = 0
    for ordered in (False, True) if "pcc" in opts else (False,):
        if ordered:
            ref.spin[:] = 0
            lat.set_spins(ref.spin)
        for n in (1, 2):
            lat.sweep(n)
            got, want = lat.observables(), ref.run(n)
            assert_obs_equal(got, want)
            if opts.get("csize"):
                np.testing.assert_array_equal(got["csize2"], want["csize2"])
            np.testing.assert_array_equal(lat.spins(), ref.spin)
            np.testing.assert_array_equal(lat.labels(), ref.label)
            np.testing.assert_array_equal(lat.bonds(), ref.bond)
            spans += int(want["spans_x"].sum() + want["spans_y"].sum())
    assert spans or "pcc" not in opts


def _ising(sw, orc, L, opts, tile_h):
    rest = {k: v for k, v in opts.items() if k != "pcc"}
    if "pcc" in opts:
        with sw.Lattice(L, seed=L, pcc=True, tile_h=tile_h, **rest) as lat:
            _check(lat, orc.pcc_chain(L, L, **rest), opts)
    else:
        with sw.Lattice(L, T=2.269185, seed=L, tile_h=tile_h, **rest) as lat:
            _check(lat, orc.sw_chain(L, 1.0, 2.269185, L, **rest), opts)


# at most 152 tiles of 32 rows: sub-tiles of 8 rows; at most 912: of 16; more: of 32
@pytest.mark.parametrize("opts", [{}, {"csize": True, "open": True}, {"pcc": True}, {"pcc": True, "csize": True},
                                  {"wind": True}, {"wind": True, "csize": True, "pcc": True}])
@pytest.mark.parametrize("L", [609, 801, 1939])
def test_rows_of_subtiles_oracle(sw, orc, L, opts):
    _ising(sw, orc, L, opts, 32)


@pytest.mark.parametrize("L,opts", [(384, {"wind": True}), (385, {"wind": True}), (1056, {"wind": True, "csize": True}),
                                    (1057, {"wind": True, "csize": True}), (1537, {"pcc": True}), (1921, {})])
def test_default_heights_oracle(sw, orc, L, opts):
    _ising(sw, orc, L, opts, 0)


# Potts tiles: 32 warps up to 101 tiles, 16 up to 304 in 2D and 608 in 3D, then 8
@pytest.mark.parametrize("opts", [{}, {"csize": True, "open": True}, {"wind": True}, {"wind": True, "csize": True}])
@pytest.mark.parametrize("dim,L", [(2, 300), (2, 1290), (2, 1681), (3, 50), (3, 97), (3, 161)])
def test_potts_pcc_warps_oracle(sw, orc, dim, L, opts):
    with sw.PottsLattice(dim, L, 2, seed=3, pcc=True, **opts) as lat:
        _check(lat, orc.PottsChain(dim, L, 2, 1.0, 1.0, 3, pcc=True, **opts), dict(opts, pcc=True))

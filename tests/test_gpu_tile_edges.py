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

"""Profiling mode times the kernels that the same calls run without it."""
import numpy as np
import pytest

import bench

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sw():
    import __graft_entry__
    __graft_entry__.build()
    from paper_0808_2109_gb300 import swgpu
    swgpu.lib()
    return swgpu


@pytest.mark.parametrize("opts", [{}, {"open": True}])
@pytest.mark.parametrize("L", [30, 64, 128])
def test_one_tile_lattice(sw, L, opts):
    torch = pytest.importorskip("torch")
    n = 4100   # more than one launch holds
    stream = torch.cuda.Stream()
    e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    with sw.Lattice(L, T=2.269185, seed=L, **opts) as ref, sw.Lattice(L, T=2.269185, seed=L, **opts) as lat:
        ref.set_stream(stream)
        ref.sweep(n)
        ref.sync()
        e0.record(stream)
        ref.sweep(n)
        e1.record(stream)
        torch.cuda.synchronize()
        lat.profile(True)
        lat.sweep(n)
        lat.profile_read()
        lat.sweep(n)
        st = lat.profile_read()
        assert st["tile_launches"] == 2 == bench.launches_of_call(L, 128, n) and st["merge_groups"] == 0
        # the same kernels: their time, give or take the clock (the tile and merge
        # kernels of such a lattice take 1.5 to 4 times as long)
        assert st["merge_ms"] == 0.0
        assert st["tile_ms"] == pytest.approx(e0.elapsed_time(e1), rel=0.2)
        assert lat.observables().tobytes() == ref.observables().tobytes()
        np.testing.assert_array_equal(lat.spins(), ref.spins())
        np.testing.assert_array_equal(lat.labels(), ref.labels())
        np.testing.assert_array_equal(lat.bonds(), ref.bonds())


@pytest.mark.parametrize("L,opts", [(129, {}), (64, {"csize": True}), (64, {"wind": True})])
def test_tiles_and_merges(sw, L, opts):
    with sw.Lattice(L, T=2.269185, seed=1, **opts) as lat:
        lat.profile(True)
        lat.sweep(5)
        st = lat.profile_read()
        assert st["tile_launches"] == st["merge_groups"] == 6
        assert st["tile_ms"] > 0.0 and st["merge_ms"] > 0.0
        lat.sweep(2)
        assert lat.profile_read()["tile_launches"] == 3

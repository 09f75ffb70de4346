"""A server's failures, injected on the host (no GPU fault), and its memory
budget: a job ends with the error that kept it from running, the jobs beside it
run on, and no device memory of the jobs goes uncounted."""
import time

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


def _run_one(sw, srv, orc, seed):
    (i,) = srv.submit([{"L": 70, "T": 2.3, "sweeps": 4, "seed": seed, "tile_h": 64}], want_spins=True)
    srv.wait_all(60.0)
    res, out = srv.poll(i)
    ref = orc.sw_chain(70, 1.0, 2.3, seed)
    assert res.status == 0
    assert_obs_equal(out["obs"], ref.run(4))
    np.testing.assert_array_equal(out["spins"], ref.spin)


@pytest.mark.parametrize("opts", [{"T": 2.3}, {"pcc": True}, {"T": 2.3, "csize": True, "wind": True}])
@pytest.mark.parametrize("jobs", [1, 3])
def test_failed_setup_ends_its_jobs(sw, orc, jobs, opts):
    with sw.Server() as srv:
        sw.sw_debug_fail_setups(1)
        try:
            ids = srv.submit([dict(opts, L=200, sweeps=30, seed=r, tile_h=64) for r in range(jobs)])
            srv.wait_all(60.0)
        finally:
            sw.sw_debug_fail_setups(0)
        for i in ids:
            res, out = srv.poll(i)
            assert res.status == sw.SW_ERR_CUDA
            assert out["obs"].tobytes() == bytes(out["obs"].nbytes)   # nothing ran
        st = srv.stats()
        assert st["bytes_in_use"] == 0 and st["active"] == 0 and st["finished"] == jobs
        _run_one(sw, srv, orc, 5)


def test_failed_setup_leaves_other_jobs_alone(sw, orc):
    """Two lanes get jobs together and the second one's set-up fails; then jobs join
    a lane whose other job runs on."""
    with sw.Server() as srv:
        sw.sw_debug_fail_setups(1, skip=1)
        try:
            good, bad = srv.submit([{"L": 96, "T": 2.3, "sweeps": 6, "seed": 1, "tile_h": 32},
                                    {"L": 96, "T": 2.3, "sweeps": 6, "seed": 1, "tile_h": 96}])
            srv.wait_all(60.0)
        finally:
            sw.sw_debug_fail_setups(0)
        assert srv.poll(bad)[0].status == sw.SW_ERR_CUDA
        res, out = srv.poll(good)
        assert res.status == 0
        assert_obs_equal(out["obs"], orc.sw_chain(96, 1.0, 2.3, 1).run(6))

        (first,) = srv.submit([{"L": 512, "T": 2.3, "sweeps": 4000, "seed": 9, "tile_h": 64}], want_spins=True)
        while srv.stats()["active"] == 0:
            time.sleep(0.001)
        sw.sw_debug_fail_setups(1)
        try:
            late = srv.submit([{"L": 128, "T": 2.3, "sweeps": 6, "seed": r, "tile_h": 64} for r in range(2)])
            srv.wait_all(60.0)
        finally:
            sw.sw_debug_fail_setups(0)
        assert [srv.poll(i)[0].status for i in late] == [sw.SW_ERR_CUDA] * 2
        res, out = srv.poll(first)
        assert res.status == 0
        with sw.Lattice(512, T=2.3, seed=9) as lat:
            lat.sweep(4000)
            assert_obs_equal(out["obs"], lat.observables())
            np.testing.assert_array_equal(out["spins"], lat.spins())
        _run_one(sw, srv, orc, 6)


def _bytes_in_use(sw, srv, specs):
    """The budget's bytes that these jobs take together, once all of them run."""
    ids = srv.submit(specs)
    deadline = time.time() + 60
    while srv.stats()["active"] < len(specs) and time.time() < deadline:
        time.sleep(0.001)
    return ids, srv.stats()["bytes_in_use"]


def test_shared_block_stays_charged_until_its_last_job(sw, orc):
    """Jobs of one lane and length share a block.  One of them fails at its
    admission: the block stays, and so do its bytes."""
    spec = {"L": 300, "T": 2.3, "sweeps": 6000, "tile_h": 96}
    with sw.Server() as srv:
        _, two = _bytes_in_use(sw, srv, [dict(spec, seed=r) for r in range(2)])
        srv.wait_all(60.0)
        sw.sw_debug_fail_allocations(1)
        try:
            bad, good = srv.submit([dict(spec, seed=1), dict(spec, seed=2)], want_spins=True)
            while (got := srv.poll(bad)) is None:
                time.sleep(0.001)
        finally:
            sw.sw_debug_fail_allocations(0)
        assert got[0].status == sw.SW_ERR_NOMEM
        held = srv.stats()["bytes_in_use"]
        assert srv.poll(good) is None   # still running
        assert held == two
        srv.wait_all(60.0)
        res, out = srv.poll(good)
        assert res.status == 0
        with sw.Lattice(300, T=2.3, seed=2) as lat:
            lat.sweep(6000)
            assert_obs_equal(out["obs"], lat.observables())
            np.testing.assert_array_equal(out["spins"], lat.spins())
        assert srv.stats()["bytes_in_use"] == 0


def test_workspaces_stay_inside_the_budget(sw, orc):
    """Jobs that fill the budget leave nothing for the tables that gather their
    results (64 MiB here): the server then holds no device memory beside them once
    they are done.  With room left it keeps them, until a job needs that room."""
    import torch
    specs = [{"L": 3, "T": 2.3, "sweeps": 6000, "seed": r, "tile_h": 32} for r in range(128)]
    with sw.Server() as srv:
        _, total = _bytes_in_use(sw, srv, specs)
        srv.wait_all(120.0)

    def run(budget):
        srv = sw.Server(device_bytes=budget)
        ids = srv.submit(specs)
        srv.wait_all(120.0)
        for r in (0, 77, 127):
            res, out = srv.poll(ids[r])
            assert res.status == 0
            assert_obs_equal(out["obs"], orc.sw_chain(3, 1.0, 2.3, r).run(6000))
        return srv

    def held(srv):
        """Device bytes that the server itself gives back (the jobs' blocks stay in
        the allocator's pool)."""
        torch.cuda.synchronize()
        free0, _ = torch.cuda.mem_get_info()
        srv.close()
        return torch.cuda.mem_get_info()[0] - free0

    assert held(run(total)) < 48 << 20
    srv = run(4 * total)   # the workspace is kept ...
    (i,) = srv.submit([{"L": 3, "T": 2.3, "sweeps": int(3.9 * 128 * 6000), "seed": 1, "tile_h": 32}])
    while srv.stats()["pending"]:
        time.sleep(0.001)
    assert srv.stats()["bytes_in_use"] + (64 << 20) > 4 * total
    assert held(srv) < 48 << 20   # ... and given back for a job that needs all of the budget

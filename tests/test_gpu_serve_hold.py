"""A lone small request waits for company while a batch runs, but for microseconds: neither a long batch
nor a long poll interval of the caller's keeps it from a free slot."""
import time

import pytest

import scenegen

pytestmark = pytest.mark.gpu


def test_small_request_beside_a_long_batch():
    import paper_2405_13364_gb300 as P
    # lists of hundreds of thousands of references: more than 5 ms
    long_scene = P.DeviceScene.from_scene(scenegen.gaussian_particles(1_000_000, 200, 100, seed=1))
    small = P.DeviceScene.from_scene(scenegen.frustum_parallelograms(500, 64, 64, seed=2))
    srv = P.Server(num_slots=2, max_batch_views=4, slot_workspace_bytes=512 << 20, poll_interval_us=200_000)
    for s, size in ((long_scene, (200, 100)), (small, (64, 64))):       # kernels loaded
        assert srv.poll(srv.submit(s, *size), timeout_us=5_000_000)[0] == 0
    waits = []
    for _ in range(5):
        before, end = srv.stats()["batches"], time.time() + 5
        t_long = srv.submit(long_scene, 200, 100)
        while srv.stats()["batches"] == before and time.time() < end:    # until it runs, the other slot free
            pass
        t_small = srv.submit(small, 64, 64)
        big = srv.poll(t_long, timeout_us=5_000_000)
        got = srv.poll(t_small, timeout_us=5_000_000)
        assert big[0] == 0 and got[0] == 0
        assert big[2]["done_ns"] - big[2]["launch_ns"] > 5_000_000
        assert got[2]["batch_views"] == 1
        waits.append(got[2]["launch_ns"] - got[2]["submit_ns"])
    srv.close()
    # 40 us of waiting; the rest is the launch itself and what the host's scheduler takes
    assert sorted(waits)[2] < 1_000_000, waits

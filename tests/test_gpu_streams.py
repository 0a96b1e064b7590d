"""Other streams beside a solve: a solve in one thread, small kernels on a stream of
their own in another.  Alone such a kernel takes some ten microseconds; beside a
solve it may wait for the launch that holds the SMs, but not for the whole solve.
The times are compared with the solve's own, with wide margins."""
import threading
import time

import pytest

import hp_synth
from gpu_util import need_gpu, torch

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]


def _beside(kw, seconds):
    """Latencies (ms) of small kernels while solves run, and the step loop's time (ms)."""
    need_gpu()
    import paper_2301_04642_gb300 as fe
    c = fe.Context(device=0)
    for _ in range(2):
        c.solve(**kw)
    loop = c.phase_ms()["loop_ms"]
    s, x, lat, errors = torch.cuda.Stream(), torch.randn(500, 500, device="cuda"), [], []
    stop = time.time() + seconds

    def solves():
        try:
            while time.time() < stop:
                c.solve(**kw)
        except Exception as e:
            errors.append(e)

    t = threading.Thread(target=solves)
    t.start()
    while time.time() < stop:
        a = time.perf_counter()
        with torch.cuda.stream(s):
            x * 2.0
        s.synchronize()
        lat.append((time.perf_counter() - a) * 1e3)
    t.join()
    c.close()
    assert not errors
    return sorted(lat), loop


def test_small_solve_leaves_the_other_sms():
    """n = 517 at finite temperature: 27 tiles, 54 of 152 SMs."""
    p = hp_synth.smeared(517, 440, 0.01, -2.0, 1.0, 7100)
    lat, loop = _beside(dict(H=torch.from_numpy(p.H).cuda(), ne=440, kT=0.01), 2.0)
    print(len(lat), lat[int(0.95 * len(lat))], lat[-1], loop)
    assert lat[int(0.95 * len(lat))] < 0.25 * loop


def test_large_solve_lets_other_streams_in():
    """n = 4096 at finite temperature: about 130 steps of a fifth of a millisecond on
    every SM."""
    n, ne = 4096, 3500
    p = hp_synth.smeared_reflected(n, ne, 0.01, -2.0, 1.0, 7200, device="cuda")
    lat, loop = _beside(dict(H=p.H, ne=ne, kT=0.01), 3.0)
    print(len(lat), lat[int(0.99 * len(lat))], lat[-1], loop)
    assert lat[int(0.99 * len(lat))] < 0.6 * loop


def test_served_request_beside_blocking_solves():
    """A request of n = 300 on the same context, beside finite-temperature solves of n =
    4096: some three turns of the SMs for its set-up, one per eight steps and two for
    its polish, about ten turns of a third of the blocking solve each."""
    need_gpu()
    import paper_2301_04642_gb300 as fe
    n, ne = 4096, 3500
    p = hp_synth.smeared_reflected(n, ne, 0.01, -2.0, 1.0, 7200, device="cuda")
    q = hp_synth.gapped(300, 240, (-3.0, -0.05), (0.05, 1.0), 7300)
    Hq = torch.from_numpy(q.H).cuda()
    D = [torch.empty_like(Hq) for _ in range(2)]
    with fe.Context(device=0) as c:
        for _ in range(2):
            c.solve(p.H, ne, kT=0.01)
        loop = c.phase_ms()["loop_ms"]
        c.solve(Hq, 240, D=D[0])
        c.wait(c.submit(Hq, 240, D=D[1]))
        stop, errors, lat = time.time() + 3.0, [], []

        def solves():
            try:
                while time.time() < stop:
                    c.solve(p.H, ne, kT=0.01)
            except Exception as e:
                errors.append(e)

        t = threading.Thread(target=solves)
        t.start()
        while time.time() < stop:
            a = time.perf_counter()
            r = c.wait(c.submit(Hq, 240, D=D[1]), timeout_s=60)
            lat.append((time.perf_counter() - a) * 1e3)
            assert r["rc"] == 0
        t.join()
    assert not errors and float((D[0] - D[1]).norm()) <= 1e-6 * 240 ** 0.5
    lat.sort()
    print(len(lat), lat[len(lat) // 2], lat[-1], loop)
    assert lat[len(lat) // 2] < 10 / 3 * loop

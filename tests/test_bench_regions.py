"""CPU tests of the benchmark's timed regions: the default length, and that no
region of a default run passes the steps at which the sheared cell inverts."""
import sys
import types

import bench


def regions(K, repeats, done):
    """Steps from rest at which each timed region ends, and the restarts."""
    now, ends, restarts = [done], [], []

    class P:
        cf_synchronize = staticmethod(lambda ctx: None)

        @staticmethod
        def cf_step_async(ctx, n):
            now[0] += n
            ends.append(now[0])

    event = types.SimpleNamespace(record=lambda s: None, elapsed_time=lambda o: 1.0)
    cuda = types.SimpleNamespace(synchronize=lambda d: None, Event=lambda enable_timing: event)

    def restart():
        restarts.append(len(ends))
        now[0] = 200
        return 200

    ms = bench.timed_regions(P, types.SimpleNamespace(cuda=cuda), None, None, 0, K, repeats, 1, lambda: None, done, restart)
    assert len(ms) == len(ends) == repeats
    return ends, restarts


def test_default_run(monkeypatch):
    monkeypatch.setattr(sys, "argv", ["bench.py"])
    args = bench.parse()
    assert (args.steps, args.warmup, args.gpus, args.workload) == (20000, 200, 1, "shear")
    ends, restarts = regions(args.steps, args.repeats, args.warmup + 32 * args.autotune_steps)
    assert max(ends) <= bench.RESTART_STEPS < 36000 and restarts == [1, 2, 3, 4]
    assert ends[-1] + args.profile_steps + args.e2e_steps < 36000


def test_short_regions_go_on():
    ends, restarts = regions(20, 5, 1480)
    assert restarts == [] and ends == [1500, 1520, 1540, 1560, 1580]


def test_long_regions_each_start_over():
    assert regions(40000, 3, 1480) == ([41480, 40200, 40200], [1, 2])

"""CUDA-graph replay of the LSERK step sequence: identical bits to launching every kernel, for the
FP64 and FP32-bulk forms, with shock capturing, across changes of U and dt (recapture), and
interleaved with single steps; plus the time per step of the launch-bound N = 3, 4^3 workload."""
import time

import numpy as np
import pytest

from paper_2306_12891_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    from paper_2306_12891_gb300 import build, dg

    assert torch.cuda.is_available(), "GPU tests need CUDA"
    build.build()
    dg.lib()
    return dg, torch


@pytest.mark.parametrize("name,extra", [("tgv_euler_n3_4x4x4", {}),
                                        ("tgv_ns_n7_32x32x32_curved", dict(precision="fp32_bulk", p_ref=1 / 1.4e-2)),
                                        ("tgv_euler_n3_4x4x4", dict(shock_capturing=True))])
def test_graph_replay_is_bit_identical(env, name, extra):
    """(the third case runs the indicator and the DG/FV blend inside the graph)"""
    dg, torch = env
    w = W.WORKLOADS[name]
    if "shock_capturing" in extra:
        w = w.with_(shock_capturing=True)
        extra = {}
    if w.n_elems > 64:
        w = w.with_(nel=(4, 4, 4))
    xyz, faces = w.mesh()
    U0 = torch.from_numpy(w.initial_state(xyz)).cuda()
    out = []
    for graphs in (False, True):
        s = dg.DG(w.N, xyz, faces, **extra, **w.physics())
        s.use_graphs(graphs)
        dt = s.max_dt(U0, w.cfl)
        U = U0.clone()
        l0 = s.launch_count()
        s.lserk_steps(U, dt, 7)
        s.lserk_step(U, dt)              # a single step between replays
        s.lserk_steps(U, 0.5 * dt, 4)     # new dt: recapture
        V = U.clone()
        s.lserk_steps(V, dt, 3)           # new U: recapture
        s.check()
        out.append((U.clone(), V.clone(), s.launch_count() - l0))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert out[0][2] == out[1][2]


def test_small_case_time_per_step(env):
    dg, torch = env
    w = W.WORKLOADS["tgv_euler_n3_4x4x4"]
    xyz, faces = w.mesh()
    U = torch.from_numpy(w.initial_state(xyz)).cuda()
    res = {}
    for graphs in (False, True):
        s = dg.DG(w.N, xyz, faces, **w.physics())
        s.use_graphs(graphs)
        dt = s.max_dt(U, w.cfl)
        s.lserk_steps(U.clone(), dt, 10)
        V = U.clone()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        s.lserk_steps(V, dt, 1000)
        torch.cuda.synchronize()
        res[graphs] = (time.perf_counter() - t0) / 1000 * 1e6
    print(f"GRAPHS N=3 4^3 Euler: {res[False]:.1f} us/step launched, {res[True]:.1f} us/step replayed "
          f"(x{res[False] / res[True]:.2f})")
    assert res[True] < res[False]


def _small(dg, torch):
    w = W.WORKLOADS["tgv_euler_n3_4x4x4"]
    xyz, faces = w.mesh()
    s = dg.DG(w.N, xyz, faces, **w.physics())
    U = torch.from_numpy(w.initial_state(xyz)).cuda()
    return s, U, s.max_dt(U, w.cfl)


@pytest.mark.parametrize("calls", [[40, 3, 33, 16, 50], [10] * 6, [2, 100], [17, 17, 17, 5], [16, 16, 16, 16, 1],
                                   [33], [32, 1, 16], [50, 50, 2, 2, 2, 50], [9, 9, 25, 25, 9], [1, 1, 1, 20, 20]])
def test_sequences_of_calls_are_bit_identical(env, calls):
    """Calls that launch, capture, replay and mix the three give the bits and the launch count of launching every kernel."""
    dg, torch = env
    out = []
    for graphs in (False, True):
        s, U0, dt = _small(dg, torch)
        s.use_graphs(graphs)
        U, l0 = U0.clone(), s.launch_count()
        for k in calls:
            s.lserk_steps(U, dt, k)
        s.check()
        out.append((U, s.launch_count() - l0))
    assert torch.equal(out[0][0], out[1][0])
    assert out[0][1] == out[1][1]


def test_a_new_step_size_before_every_few_steps_captures_nothing(env):
    """Host time of a call of 10 steps, a new dt each time: a graph for it would be replayed once (or, of 16 steps, not at
    all), so the call costs what it costs with graphs off."""
    dg, torch = env
    cost = {}
    for graphs in (False, True):
        s, U, dt = _small(dg, torch)
        s.use_graphs(graphs)
        times = []
        for k in range(30):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            s.lserk_steps(U, dt * (1 + 1e-9 * k), 10)
            times.append(time.perf_counter() - t0)
        cost[graphs] = sorted(times)[15] * 1e6
    print(f"GRAPHS host time of 10 steps with a new dt: {cost[False]:.0f} us off, {cost[True]:.0f} us on")
    assert cost[True] < 1.3 * cost[False]


def test_a_short_first_call_does_not_shorten_the_graph(env):
    """1600 steps after a first call of 2 take what they take without it (one-step graphs: a gap at every step)."""
    dg, torch = env
    res = {}
    for first in (0, 2):
        s, U, dt = _small(dg, torch)
        dt *= 0.01
        if first:
            s.lserk_steps(U, dt, first)
        s.lserk_steps(U, dt, 100)
        times = []
        for _ in range(3):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            s.lserk_steps(U, dt, 1600)
            torch.cuda.synchronize()
            times.append((time.perf_counter() - t0) / 1600 * 1e6)
        res[first] = min(times)
    print(f"GRAPHS us/step after a first call of 0 and 2 steps: {res[0]:.2f} {res[2]:.2f}")
    assert res[2] < 1.025 * res[0]  # (one-step graphs: 1.045)

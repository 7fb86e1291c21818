"""The signed distance's wide grid, built by the first large call on an obstacle
set, beside other streams: the call waits for nothing on the host, a capture
that some thread has begun elsewhere stays valid, and calls on other streams,
capturing ones among them, are right while the build is still queued. Values
against small calls on a set of its own (no wide grid), within the 1e-6 m of
two roundings of the same expression."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
N = 20_000


@pytest.fixture()
def scene():
    import torch

    from paper_2504_10783_gb300 import ezo
    from paper_2504_10783_gb300 import workloads as wl
    rd, obs = wl.dh7_robot(), wl.box_obstacles(5, 100).spheres
    robot = ezo.Robot(rd)
    q = torch.from_numpy(np.ascontiguousarray(wl.uniform_configs(2, rd, N).astype(np.float32).T)).cuda()
    want, ref = torch.empty(N, device="cuda"), ezo.Env(obs)
    for i in range(0, N, 10_000):
        ezo.signed_distance(robot, ref, q[:, i:i + 10_000], want[i:i + 10_000])
    torch.cuda.synchronize()
    return lambda: ezo.Env(obs), (lambda env, out, s: ezo.signed_distance(robot, env, q, out, stream=s)), want


@pytest.mark.parametrize("where", ["same thread", "other thread"])
def test_first_large_call_beside_a_capture(scene, where):
    import torch
    make, call, want = scene
    env, out, other = make(), torch.zeros(N, device="cuda"), torch.cuda.Stream()
    x = torch.zeros(64, device="cuda")
    torch.cuda.synchronize()
    graph, failed = torch.cuda.CUDAGraph(), []

    def body():
        try:
            call(env, out, other)
        except Exception as e:  # noqa: BLE001
            failed.append(e)

    with torch.cuda.stream(torch.cuda.Stream()):
        graph.capture_begin(capture_error_mode="global")
        x.add_(1)
        if where == "same thread":
            body()
        else:
            t = threading.Thread(target=body)
            t.start()
            t.join()
        graph.capture_end()
        graph.replay()
    torch.cuda.synchronize()
    assert not failed and float(x[0]) == 1.0
    assert (out - want).abs().max().item() <= 1e-6


def test_queued_build_across_streams(scene):
    import torch
    make, call, want = scene
    env = make()
    first, second, third = (torch.cuda.Stream() for _ in range(3))
    outs = [torch.zeros(N, device="cuda") for _ in range(4)]
    call(make(), outs[0], first)  # kernels and their attributes loaded
    torch.cuda.synchronize()
    with torch.cuda.stream(first):
        torch.cuda._sleep(400_000_000)  # a fifth of a second of earlier work
    call(env, outs[0], first)
    assert not first.query()  # the call did not wait for it
    call(env, outs[1], second)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(third):
        graph.capture_begin(capture_error_mode="thread_local")
        call(env, outs[2], third)
        graph.capture_end()
        assert not first.query()  # the build was still queued
        graph.replay()
    torch.cuda.synchronize()
    call(env, outs[3], second)
    torch.cuda.synchronize()
    for k, out in enumerate(outs):
        assert (out - want).abs().max().item() <= 1e-6, k

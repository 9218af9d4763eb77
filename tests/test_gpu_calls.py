"""What calls need around them and leave behind: device memory, other host threads' calls, stream capture."""
import threading
import time

import numpy as np
import pytest

import graphgen as gg
from oracle import deco_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2509_18612_gb300 as deco  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("precision", [deco.DECO_PREC_FP32, deco.DECO_PREC_BF16])
def test_batches_leave_no_device_memory_behind(precision):
    # the members' images of the row-vector form (some 0.6 MiB here) are kept with the batch and go with it
    members = [deco.graph_from(gg.ba_graph(900, 4, i)) for i in range(20)]
    pop = deco.population(candidates=2, rounds=1, t_lo=1, t_hi=2, e_lo=-2.5, e_hi=-1.5, lifts=(1,))

    def program(times):
        for _ in range(times):
            b = deco.deco_create_batch(members)
            deco.deco_solve_batch(b, 16, deco.params(init=deco.DECO_INIT_IDI, precision=precision), pop, 1)
            deco.deco_destroy_batch(b)
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    before = program(3)
    assert before - program(40) <= 8 << 20


def _greedy(n):
    G = deco.graph_from(gg.er_graph_avg_degree(n, 5.0, 1))
    z, cuts = torch.zeros(n, dtype=torch.uint8, device=DEV), torch.zeros(1, dtype=torch.int64, device=DEV)
    return lambda st: deco.deco_greedy(G, 1, 1, z, cuts, stream=st)


def _search(n):
    G = deco.graph_from(gg.torus_graph(n // 4, 4, 1))
    z, cuts = torch.zeros(n * 8, dtype=torch.uint8, device=DEV), torch.zeros(8, dtype=torch.int64, device=DEV)
    return lambda st: deco.deco_local_search(G, 8, z, 1, cuts, stream=st)


def _phase(n, kernel, per_column):
    G = deco.graph_from(gg.er_graph_avg_degree(n, 5.0, 1))
    y = torch.zeros(n, 64, device=DEV)
    alpha = torch.full((64,), 0.01, device=DEV)
    args = deco.step_args(alpha_cols=alpha if per_column else None)
    return lambda st, _alpha=alpha: deco.deco_run_phase(G, 64, 64, y, None, 1, args, kernel, stream=st)


def _infer(hidden):
    G = deco.graph_from(gg.er_graph_avg_degree(500, 5.0, 1))
    m, h = deco.Mpnn(hidden, 1, 1), torch.zeros(500, device=DEV)
    return lambda st: m.infer(G, h, 1, stream=st)


def _train(hidden):
    G = deco.graph_from(gg.er_graph_avg_degree(500, 5.0, 1))
    m, z = deco.Mpnn(hidden, 1, 1), torch.zeros(500, dtype=torch.uint8, device=DEV)
    return lambda st: m.train(G, z, 1, stream=st)


SLAB = deco.DECO_KERNEL_ONCHIP | (8 << 8) | deco.DECO_KERNEL_ROW_PAIRS


# Two host threads on graphs of different sizes, each with a stream of its own: launches of the same kernels with much
# and with little shared memory in turn, none of which may refuse the other's.
@pytest.mark.parametrize("name,big,small", [
    ("greedy", lambda: _greedy(150000), lambda: _greedy(64)),
    ("search", lambda: _search(20000), lambda: _search(64)),
    ("rows", lambda: _phase(1500, deco.DECO_KERNEL_AUTO, True), lambda: _phase(40, deco.DECO_KERNEL_AUTO, True)),
    ("registers", lambda: _phase(500, deco.DECO_KERNEL_AUTO, False), lambda: _phase(300, deco.DECO_KERNEL_AUTO, False)),
    ("slab", lambda: _phase(1200, SLAB, False), lambda: _phase(60, SLAB, False)),
    ("infer", lambda: _infer(128), lambda: _infer(64)),
    ("train", lambda: _train(128), lambda: _train(64)),
])
def test_host_threads_do_not_refuse_each_others_launches(name, big, small):
    calls, errors = [big(), small()], []
    end = time.time() + 1.5

    def loop(call):
        stream = torch.cuda.Stream()
        try:
            while time.time() < end and not errors:
                for _ in range(8):
                    call(stream.cuda_stream)
                stream.synchronize()
        except deco.DecoError as e:
            errors.append(str(e))

    torch.cuda.synchronize()
    threads = [threading.Thread(target=loop, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors


# A phase whose first call on a graph, or first call of its width, is captured: the images of the on-chip forms, which
# need an allocation, are not there.  (ONCHIP: warmed with another width, whose image serves.)
@pytest.mark.parametrize("n,degree,warm,C,kernel", [
    (3000, 6.0, 0, 64, deco.DECO_KERNEL_AUTO), (800, 5.0, 0, 64, deco.DECO_KERNEL_AUTO),
    (800, 48.0, 64, 1024, deco.DECO_KERNEL_AUTO), (800, 5.0, 64, 1024, deco.DECO_KERNEL_AUTO),
    (800, 5.0, 64, 1024, deco.DECO_KERNEL_ONCHIP), (800, 5.0, 64, 64, deco.DECO_KERNEL_ONCHIP)])
@pytest.mark.parametrize("precision", [deco.DECO_PREC_FP32, deco.DECO_PREC_BF16])
def test_phases_captured_before_their_images_are_built(n, degree, warm, C, kernel, precision):
    G = deco.graph_from(gg.er_graph_avg_degree(n, degree, 1))
    dtype = torch.bfloat16 if precision else torch.float32
    args = deco.step_args(0, precision, 0.01, 0.9)
    y0 = (torch.rand(n, C, device=DEV) - 0.5).to(dtype)
    y, v = y0.clone(), torch.zeros(n, C, device=DEV)
    ref, vref = y0.clone(), v.clone()
    deco.deco_run_phase(G, C, C, ref, vref, 5, args, deco.DECO_KERNEL_GLOBAL)
    if warm:
        deco.deco_run_phase(G, warm, warm, torch.zeros(n, warm, device=DEV, dtype=dtype),
                            torch.zeros(n, warm, device=DEV), 2, args, kernel)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        deco.deco_run_phase(G, C, C, y, v, 5, args, kernel, stream=torch.cuda.current_stream().cuda_stream)
    for _ in range(2):
        y.copy_(y0)
        v.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, ref) and torch.equal(v, vref)


# What a call uploads for its first launch (the graph's arrays, an image of its rows) is there for a stream that does not
# wait for the default one.
@pytest.mark.parametrize("n,degree,C,kernel", [
    (800, 5.0, 64, deco.DECO_KERNEL_ONCHIP), (800, 48.0, 64, deco.DECO_KERNEL_AUTO),
    (1200, 5.0, 64, SLAB), (30000, 40.0, 8, deco.DECO_KERNEL_GLOBAL), (30000, 12.0, 64, deco.DECO_KERNEL_AUTO)])
def test_first_phase_on_a_non_blocking_stream(n, degree, C, kernel):
    edges = gg.er_graph_avg_degree(n, degree, 1)
    args = deco.step_args(0, deco.DECO_PREC_FP32, 0.01, 0.9)
    y0 = torch.rand(n, C, device=DEV) - 0.5
    ref, vref = y0.clone(), torch.zeros(n, C, device=DEV)
    G = deco.graph_from(edges)
    torch.cuda.synchronize()
    deco.deco_run_phase(G, C, C, ref, vref, 5, args, deco.DECO_KERNEL_GLOBAL)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    for _ in range(5):
        y, v = y0.clone(), torch.zeros(n, C, device=DEV)
        torch.cuda.synchronize()
        first = deco.graph_from(edges)   # held until the stream has run
        deco.deco_run_phase(first, C, C, y, v, 5, args, kernel, stream=stream.cuda_stream)
        stream.synchronize()
        assert torch.equal(y, ref) and torch.equal(v, vref)

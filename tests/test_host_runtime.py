"""The library's host code (planning, graphs, the small-step schedule) without a GPU: libtn.so's
object files linked against a stand-in for the CUDA runtime (fake_cudart.c), whose kernels do
nothing.  Each test runs in a process of its own."""
import os
import re
import shutil
import subprocess
import sys
import textwrap

import pytest

from paper_2310_03978_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = """
import ctypes as C, sys, types
import numpy as np
from paper_2310_03978_gb300 import tn, workload as W
tn.LIB_PATH = sys.argv[1]
L = tn.lib()
L.fake_calls.restype = L.fake_alive.restype = C.c_long
calls = lambda name: L.fake_calls(name.encode())
NULL = types.SimpleNamespace(cuda_stream=0)
MINE = types.SimpleNamespace(cuda_stream=64)

def net_of(labels, opens):
    return tn.Network([np.zeros((2,) * len(l), complex) for l in labels], labels, opens)
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    cc = shutil.which("gcc")
    if cc is None or os.uname().sysname != "Linux":
        pytest.skip("needs gcc")
    B.build()
    out = str(tmp_path_factory.mktemp("fake") / "libtn_fake.so")
    objs = [os.path.join(B.BUILD, os.path.splitext(s)[0] + ".o") for s in B.SOURCES]
    # -Bsymbolic: the stand-in serves this library only, whatever else the process has loaded
    subprocess.run([cc.replace("gcc", "g++"), "-shared", "-fPIC", "-Wl,-Bsymbolic", "-o", out,
                    "-x", "c", os.path.join(HERE, "fake_cudart.c"), "-x", "none", *objs],
                   check=True)

    def run(code):
        r = subprocess.run([sys.executable, "-c", PRELUDE + textwrap.dedent(code), out], cwd=ROOT,
                           capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, "exit %d\n%s%s" % (r.returncode, r.stdout, r.stderr)
        return r.stdout

    return run


# Connected steps on one rank-12 leaf (g: one-qubit gate, v: vector, p: a tensor of two of its labels,
# o: outer product with a vector).  Tensors, records and padding take as many complex64 as the key
# says; a block's shared memory holds 27648, so the last two work in global memory.
RUNS = {27646: "ggvvpvvvppvo", 27647: "ggvvpvvpgpvvov", 27648: "ggvvpvvvpvvv",
        27649: "ggvvpvvvpvg", 27650: "ggvvpvvvpvpo"}


def run_network(ops):
    """(labels, open labels, path) of the run."""
    wires, fresh = list(range(12)), 100
    labels, path = [list(wires)], []
    for op in ops:
        k, n = {"g": (1, 1), "v": (1, 0), "p": (2, 0), "o": (0, 1)}[op]
        cut, wires = wires[:k], wires[k:]
        new = list(range(fresh, fresh + n))
        fresh += n
        labels.append(cut + new)
        wires += new
        path.append((0, len(labels) - 1))
    return labels, wires, path


@pytest.mark.parametrize("size", RUNS)
def test_runs_of_small_steps_that_just_fit_shared_memory(fake, size):
    labels, opens, path = run_network(RUNS[size])
    fake("""
    net = net_of(%r, %r)
    plan = tn.Plan(net, %r)
    plan.contract_host(stream=NULL)
    assert calls("launch") > 0
    plan.close(); net.close()
    """ % (labels, opens, path))


# (rows, cols, cycles, open qubits, sliced bonds, mode): what one slice takes when the steps run in path
# order, in bytes.  A plan may use more to save launches, but only where the workspace allows it.
IN_PATH_ORDER = {(5, 5, 10, 6, 4, "c64"): 5081088, (5, 5, 10, 6, 4, "fp16_scaled"): 4016128,
                 (3, 5, 11, 12, 0, "tf32"): 1599488, (4, 3, 6, 12, 0, "tf32"): 81920,
                 (4, 5, 12, 10, 2, "split_tf32"): 489882624}


@pytest.mark.parametrize("case", IN_PATH_ORDER, ids=str)
def test_a_workspace_of_what_path_order_takes_is_enough(fake, case):
    fake("""
    rows, cols, cycles, opens, nsl, mode = %r
    need, q = %d, rows * cols
    net = W.build_network(W.random_circuit(rows, cols, cycles, 3), list(range(q - opens, q)),
                          {i: 0 for i in range(q - opens)})
    path = W.greedy_path(net.labels, net.open_labels)
    cut = W.greedy_slices(net.labels, net.open_labels, path, nsl) if nsl else []
    tnet = tn.Network.from_workload(net)
    for graph in (False, True):
        plan = tn.Plan(tnet, path, cut, mode=mode, use_graph=graph, max_slices_in_flight=1,
                       workspace_limit=need)
        assert plan.info()["workspace_bytes"] <= need
        plan.close()
        # and no slices in flight are lost to it
        free = tn.Plan(tnet, path, cut, mode=mode, use_graph=False)
        limit = free.info()["workspace_bytes"]
        plan = tn.Plan(tnet, path, cut, mode=mode, use_graph=graph, workspace_limit=limit)
        assert plan.info()["slices_in_flight"] == free.info()["slices_in_flight"]
        plan.close(); free.close()
    """ % (case, IN_PATH_ORDER[case]))


def test_direct_launches_on_the_default_stream_take_no_branches(fake):
    # branches of the prologue exist in a captured graph only; the default stream's handle is 0, as is
    # a stream's that has not been made yet
    fake("""
    net = W.build_network(W.random_circuit(3, 4, 8, 3), list(range(6, 12)), {i: 0 for i in range(6)})
    path = W.greedy_path(net.labels, net.open_labels)
    cut = W.greedy_slices(net.labels, net.open_labels, path, 2)
    tnet = tn.Network.from_workload(net)
    for stream in (NULL, MINE):
        plan = tn.Plan(tnet, path, cut, use_graph=True, max_slices_in_flight=1)
        plan.contract_host(0, 1, stream=stream)
        assert calls("cudaStreamWaitEvent") == 0 and calls("cudaEventRecord") == 0
        plan.close()
    # as a whole call, and again for work of up to 4 launches, which never becomes a graph
    plan = tn.Plan(tnet, path, cut, use_graph=True)
    plan.contract_host(stream=NULL)
    assert calls("cudaStreamWaitEvent") == 0
    plan.close()
    tnet.close()
    """)


@pytest.mark.parametrize("call", ["cudaGraphInstantiate", "cudaStreamBeginCapture",
                                  "cudaStreamCreateWithFlags", "cudaEventCreateWithFlags"])
def test_a_graph_that_cannot_be_made_leaves_the_direct_launches(fake, call):
    fake("""
    net = W.build_network(W.random_circuit(4, 5, 10, 3), list(range(12, 20)), {i: 0 for i in range(12)})
    path = W.greedy_path(net.labels, net.open_labels)
    cut = W.greedy_slices(net.labels, net.open_labels, path, 2)
    tnet = tn.Network.from_workload(net)
    amps = C.create_string_buffer(16 << 8)

    def sparse():
        plan = tn.SparsePlan(tnet, path, np.zeros((4, 8), np.uint8))
        run = lambda: tn._check(L.tn_sparse_contract(plan.handle, amps, C.c_void_p(64)))
        return plan, run, lambda: plan.info()["kernel_launches"]

    def dense(flight):
        plan = tn.Plan(tnet, path, cut, use_graph=True, max_slices_in_flight=flight)
        run = lambda: plan.contract_host(stream=MINE)
        return plan, run, lambda: plan.info()["kernel_launches"]

    # one slice in flight: two graphs, of which the batch's has no branches and needs no events
    for make in (sparse, lambda: dense(0), lambda: dense(1))[:2 if "%s" == "cudaEventCreateWithFlags" else 3]:
        before = [L.fake_alive(k) for k in range(5)]
        plan, run, launched = make()
        L.fake_fail(b"%s", 0, 1000)
        run()
        first = launched()
        for _ in range(2):
            run()
        L.fake_fail(b"%s", 0, 0)
        run()
        assert calls("cudaGraphLaunch") == 0 and launched() == 4 * first
        assert L.fake_alive(2) == before[2] and L.fake_alive(3) == 0
        plan.close()
        assert [L.fake_alive(k) for k in range(5)] == before
    tnet.close()
    """ % (call, call, call))


def test_a_callers_capture_takes_the_launches_themselves(fake):
    fake("""
    net = W.build_network(W.random_circuit(4, 5, 10, 3), list(range(12, 20)), {i: 0 for i in range(12)})
    path = W.greedy_path(net.labels, net.open_labels)
    cut = W.greedy_slices(net.labels, net.open_labels, path, 2)
    tnet = tn.Network.from_workload(net)
    L.fake_capture.argtypes, made = [C.c_void_p], 0
    for flight in (0, 1):
        plan = tn.Plan(tnet, path, cut, use_graph=True, max_slices_in_flight=flight)
        L.fake_capture(64)
        for _ in range(3):
            plan.contract_host(stream=MINE)
        assert calls("cudaStreamBeginCapture") == made
        L.fake_capture(0)
        plan.contract_host(stream=MINE)  # used before: now a graph
        assert calls("cudaStreamBeginCapture") > made
        made = calls("cudaStreamBeginCapture")
        plan.close()
    tnet.close()
    """)


def test_a_change_of_any_included_header_rebuilds_the_library():
    known = {os.path.basename(h) for h in B.headers()}
    for name in os.listdir(B.CSRC):
        with open(os.path.join(B.CSRC, name)) as f:
            for header in re.findall(r'#include "([^"]+)"', f.read()):
                assert os.path.basename(header) in known, "%s includes %s" % (name, header)

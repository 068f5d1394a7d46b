"""Parts of a plan that are built by the first SpMM call that needs them: first calls from several host threads on one stream, and
a first call that is captured into a graph."""
import threading

import numpy as np
import pytest
import torch

import gen
import oracle
import paper_2603_07169_b200 as b200sp
from gpu_util import assert_within, empty_out, needs_plain_build, store, to_dev, to_host

pytestmark = pytest.mark.gpu


def long_rows(m, n, k):
    """Even rows, some of them of 129-1024 nonzeros and one longer: by rows, with both lists."""
    lens = np.full(m, 9)
    lens[::500] = 150
    lens[7] = 1100
    return gen.random_csr(m, n, lens, seed=k, sort_cols=True)


# name: matrix, k, options: the lists (k-sliced kernels and the scalar ones), the shares of a large matrix, the order of the rows with B in shared memory
CASES = {
    "lists": (lambda: long_rows(30_000, 20_000, 1), 32, {"spmm_flat": 0}),
    "lists_ragged": (lambda: long_rows(30_000, 20_000, 2), 7, {"spmm_flat": 0}),
    "shares": (lambda: gen.uniform_rows(1 << 20, 1 << 18, 8, 3), 5, {"spmm_flat": 1}),
    "row_order": (lambda: long_rows(20_000, 1500, 4), 64, {}),
}


class Problem:
    def __init__(self, case, dtype="f32"):
        make, self.k, self.options = CASES[case]
        self.A, self.dtype = make(), dtype
        rng = np.random.default_rng(1)
        B, vals = store(rng.standard_normal(self.A.n * self.k).astype(np.float32), dtype), store(self.A.vals, dtype)
        self.d = [to_dev(a) for a in (self.A.row_ptr, self.A.col_idx, vals, B)]
        rows = np.unique(np.concatenate([np.arange(0, self.A.m, 97), [7, 500, self.A.m - 1]]))
        self.rows = rows
        self.ref, self.S = oracle.spmm_csr(self.A.m, self.A.n, self.k, self.A.row_ptr, self.A.col_idx, vals, B, None, 1.0, 0.0, dtype, rows=rows)
        for name, value in self.options.items():
            b200sp.b200sp_set_option(name, value)

    def close(self):
        for name in self.options:
            b200sp.b200sp_set_option(name, {"spmm_flat": 2}[name])

    def plan(self):
        return b200sp.b200sp_plan_create(self.A.m, self.A.n, self.A.nnz, self.d[0])

    def out(self):
        return empty_out(self.A.m * self.k, self.dtype)

    def call(self, plan, Y, stream=None):
        b200sp.b200sp_spmm(plan, self.k, self.d[1], self.d[2], self.d[3], Y, 1.0, 0.0, self.dtype, stream)

    def check(self, Y, what):
        assert_within(to_host(Y, self.dtype).reshape(self.A.m, self.k)[self.rows], self.ref, self.S, self.dtype, what=what)


@pytest.mark.parametrize("case", sorted(CASES))
def test_first_calls_from_several_threads(case):
    P = Problem(case)
    try:
        stream = torch.cuda.Stream()
        for trial in range(10):
            plan = P.plan()
            outs = [P.out() for _ in range(4)]
            torch.cuda.synchronize()
            barrier, failures = threading.Barrier(4), []

            def work(Y):
                try:
                    barrier.wait()
                    P.call(plan, Y, stream)
                except BaseException as e:      # noqa: BLE001 - reported below
                    failures.append(e)

            threads = [threading.Thread(target=work, args=(Y,)) for Y in outs]
            for t in threads:
                t.start()
            for t in threads:
                t.join()
            assert not failures, failures[0]
            torch.cuda.synchronize()
            P.check(outs[0], "%s trial %d" % (case, trial))
            for Y in outs[1:]:
                assert torch.equal(Y, outs[0])
            b200sp.b200sp_plan_destroy(plan)
    finally:
        P.close()


@needs_plain_build
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("case", sorted(CASES))
def test_first_call_captured(case, dtype):
    """What the captured call builds belongs to its graph: calls outside it, before it has run and after it is gone, build their own."""
    P = Problem(case, dtype)
    try:
        warm, Y = P.plan(), P.out()
        P.call(warm, Y)                         # kernels loaded, attributes set
        torch.cuda.synchronize()
        P.check(Y, "eager")
        b200sp.b200sp_plan_destroy(warm)
        plan, captured, before, after = P.plan(), P.out(), P.out(), P.out()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            P.call(plan, captured)
        P.call(plan, before)
        torch.cuda.synchronize()
        P.check(before, "outside the graph, before it has run")
        for _ in range(2):
            captured.fill_(0)
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(captured, before)
        del graph
        P.call(plan, after)
        torch.cuda.synchronize()
        assert torch.equal(after, before)
        b200sp.b200sp_plan_destroy(plan)
    finally:
        P.close()


@pytest.mark.parametrize("side_stream", [False, True])
def test_a_plan_destroyed_behind_its_product(side_stream):
    """A new pattern in every step, nothing waited for between the calls: the memory that a plan gives back is the next plan's at once, and each
    product is done with it by then."""
    P, side = Problem("lists"), torch.cuda.Stream()
    others = [gen.random_csr(20_000 + 100 * i, 20_000, np.random.default_rng(i).integers(0, 30, 20_000 + 100 * i), seed=i) for i in range(3)]
    try:
        work = [(A, [to_dev(a) for a in (A.row_ptr, A.col_idx, A.vals)], empty_out(A.m * P.k, "f32")) for A in [P.A] + others]
        torch.cuda.synchronize()
        first = None
        for step in range(40):
            outs = []
            for A, d, Y in work:
                plan = b200sp.b200sp_plan_create(A.m, A.n, A.nnz, d[0])
                b200sp.b200sp_spmm(plan, P.k, d[1], d[2], P.d[3], Y, 1.0, 0.0, "f32", side if side_stream and step % 2 else None)
                b200sp.b200sp_plan_destroy(plan)
                outs.append(Y.clone() if step in (0, 39) else None)
            if step == 0:
                first = outs
        torch.cuda.synchronize()
        P.check(work[0][2], "last step")
        assert all(torch.equal(a, b) for a, b in zip(first, outs))
    finally:
        P.close()


@pytest.mark.parametrize("side_stream", [False, True])
def test_nothing_is_in_flight_once_a_plan_is_destroyed(side_stream):
    """b200sp_plan_destroy waits for the device: from then on another stream, or the host, may read Y and reuse the operands, whichever stream the
    product ran on."""
    A, k = gen.uniform_rows(1 << 18, 1 << 18, 32, 1), 64
    d = [to_dev(a) for a in (A.row_ptr, A.col_idx, A.vals)]
    B, Y = torch.ones(A.n * k, device="cuda:0"), torch.zeros(A.m * k, device="cuda:0")
    stream, other = torch.cuda.Stream() if side_stream else torch.cuda.default_stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    in_flight = False
    for _ in range(5):
        plan = b200sp.b200sp_plan_create(A.m, A.n, A.nnz, d[0], stream)
        for _ in range(10):                                       # (1.6 ms)
            b200sp.b200sp_spmm(plan, k, d[1], d[2], B, Y, 1.0, 0.0, "f32", stream)
        in_flight |= not stream.query()
        b200sp.b200sp_plan_destroy(plan)
        assert stream.query()
        with torch.cuda.stream(other):
            copy = Y.clone()
        other.synchronize()
        assert torch.equal(copy, Y)
    assert in_flight                                              # before the call, or the rest shows nothing

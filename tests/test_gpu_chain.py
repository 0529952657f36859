"""Chained launches: a call's kernels may start before the one ahead has ended and
wait for it on the device. Tables and samples must not depend on how a call was queued:
directly, behind another call on the same stream, next to one on another stream, or by
replaying a captured graph after the input changed in place. All comparisons are
bitwise."""
import numpy as np
import pytest
import torch

import synthetic
import paper_2511_14923_gb300 as gbs

pytestmark = pytest.mark.gpu

# chunked orders only; order 4 by the tree (refined from 64 modes); order 5; no chain
TABLES = [(5, 2, "fp64"), (9, 3, "fp64"), (40, 4, "fp64"), (70, 4, "fp32r"), (30, 5, "fp64"), (41, 5, "fp32r")]


@pytest.fixture(scope="module", autouse=True)
def built():
    gbs.build()


def states(M, kmax):
    return [torch.from_numpy(synthetic.random_instance(M, kmax, seed=8100 + M + i, r_range=(0.4, 1.4)).V).cuda()
            for i in range(2)]


@pytest.mark.parametrize("M,kmax,precision", TABLES)
def test_table_from_graph_and_in_company(M, kmax, precision):
    a, b = states(M, kmax)
    ref = [gbs.cumulants(v, kmax, precision).clone() for v in (a, b)]
    # one after the other on a stream, no wait between, one workspace
    ws = gbs.Workspace(M, kmax, precision)
    outs = [torch.empty_like(ref[0]) for _ in range(4)]
    for i, o in enumerate(outs):
        gbs.cumulants((a, b)[i % 2], kmax, precision, out=o, workspace=ws, check=False)
    assert all(torch.equal(o, ref[i % 2]) for i, o in enumerate(outs)) and ws.status() == 0
    # on two streams at once
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    works = [gbs.Workspace(M, kmax, precision) for _ in streams]
    torch.cuda.synchronize()
    for rep in range(3):
        for i, s in enumerate(streams):
            with torch.cuda.stream(s):
                gbs.cumulants((a, b)[i], kmax, precision, out=outs[i], workspace=works[i], check=False)
    torch.cuda.synchronize()
    assert torch.equal(outs[0], ref[0]) and torch.equal(outs[1], ref[1])
    # captured, replayed after V changed in place
    v, out = a.clone(), torch.empty_like(ref[0])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        gbs.cumulants(v, kmax, precision, out=out, workspace=ws, check=False)
    for i in (0, 1, 0):
        v.copy_((a, b)[i])
        graph.replay()
        assert torch.equal(out, ref[i])


@pytest.mark.parametrize("K,precision,batch", [(3, "fp32", 256), (3, "fp64", 128), (4, "fp32", 128), (5, "fp32", 256),
                                               (5, "fp64", 128)])
def test_sampler_from_graph_and_in_company(K, precision, batch):
    M, n = 21, 2 * batch - 56  # two chunks, the second one ragged
    kappa = gbs.spin_cumulants(states(M, K)[0], K, "fp64")
    u = [torch.from_numpy(np.random.default_rng(31 + i).random((n, M))).cuda() for i in range(2)]
    run = lambda x, w=None: gbs.sample(kappa, M, K, u=x, batch=batch, precision=precision, workspace=w, check=False)
    ref = [[t.clone() for t in run(x)[:2]] for x in u]
    size = gbs.sampler_workspace_bytes(M, K, batch, precision)
    ws = torch.empty(size, dtype=torch.uint8, device="cuda")
    same = lambda got, want: torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    got = [run(u[i % 2], ws) for i in range(4)]
    assert all(same(g, ref[i % 2]) for i, g in enumerate(got))
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    works = [torch.empty(size, dtype=torch.uint8, device="cuda") for _ in streams]
    torch.cuda.synchronize()
    got = [None, None]
    for i, s in enumerate(streams):
        with torch.cuda.stream(s):
            got[i] = run(u[i], works[i])
    torch.cuda.synchronize()
    assert same(got[0], ref[0]) and same(got[1], ref[1])
    x = u[0].clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = run(x, ws)
    for i in (0, 1, 0):
        x.copy_(u[i])
        graph.replay()
        assert same(out, ref[i])

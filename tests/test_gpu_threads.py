"""Host threads that form tables of different sizes at once, each on a stream and in a
workspace of its own, get what each gets alone (bit for bit)."""
import ctypes
import threading

import pytest
import torch

import synthetic
import paper_2511_14923_gb300 as gbs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kmax,tops", [(3, (740, 1000)), (3, (1000, 740, 860, 940))])
def test_slices_of_different_sizes_from_several_threads(kmax, tops):
    """Chunks of orders with large top elements take more than 48 KB of shared memory,
    each top element another amount, by a limit that belongs to the kernel. One slice of
    the top order per call, through the C entry point, so that the threads' calls meet."""
    gbs.build()
    M = 1000
    V = torch.from_numpy(synthetic.random_instance(M, kmax, seed=9500, n_squeezed=8).V).cuda()
    lib, size = gbs.lib(), int(gbs.lib().gbs_range_workspace_bytes(M, kmax, 0))
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    keep, calls, outs = [], [], []
    for c in tops:
        ws = torch.empty(size, dtype=torch.uint8, device="cuda")
        out = torch.empty(gbs.range_entries(M, kmax, c - 1, c), dtype=torch.float64, device="cuda")
        s = torch.cuda.Stream()
        keep.append((ws, s))
        outs.append(out)
        calls.append((p(V), M, kmax, 2, c - 1, c, p(out), 0, p(ws), size, ctypes.c_void_p(s.cuda_stream)))
    torch.cuda.synchronize()
    want = []
    for call, out in zip(calls, outs):
        assert lib.gbs_table_range(*call) == 0
        torch.cuda.synchronize()
        want.append(out.clone())
        out.zero_()
    torch.cuda.synchronize()
    failed, start = [0] * len(calls), threading.Barrier(len(calls))

    def work(i):
        start.wait()
        for _ in range(4000):
            failed[i] += lib.gbs_table_range(*calls[i]) != 0

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(calls))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert failed == [0] * len(calls)
    assert all(torch.equal(o, w) for o, w in zip(outs, want))


def test_covariance_adjoints_of_different_sizes_from_several_threads():
    """The covariance model's adjoint takes more than 48 KB above 1536 modes, by M."""
    gbs.build()
    lib, p = gbs.lib(), lambda t: ctypes.c_void_p(t.data_ptr())
    keep, calls, outs = [], [], []
    for M in (1540, 1900, 1700):
        g = torch.Generator("cuda").manual_seed(M)
        rand = lambda *shape: torch.rand(*shape, dtype=torch.float64, device="cuda", generator=g)
        args = [rand(M, M) / M, rand(M, M) / M, rand(M), 0.2 + 0.5 * rand(M), rand(2 * M, 2 * M), rand(2 * M, 2 * M)]
        out, s = torch.zeros(2, M, dtype=torch.float64, device="cuda"), torch.cuda.Stream()
        keep.append((args, s))
        outs.append(out)
        calls.append((*map(p, args[:4]), M, *map(p, args[4:]), p(out[0]), p(out[1]), ctypes.c_void_p(s.cuda_stream)))
    torch.cuda.synchronize()
    want = []
    for call, out in zip(calls, outs):
        assert lib.gbs_covariance_backward(*call) == 0
        torch.cuda.synchronize()
        want.append(out.clone())
        out.zero_()
    torch.cuda.synchronize()
    failed, start = [0] * len(calls), threading.Barrier(len(calls))

    def work(i):
        start.wait()
        for _ in range(40):
            failed[i] += lib.gbs_covariance_backward(*calls[i]) != 0

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(calls))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert failed == [0] * len(calls)
    assert all(torch.equal(o, w) for o, w in zip(outs, want))

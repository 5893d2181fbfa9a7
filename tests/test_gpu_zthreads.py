"""Calls from several host threads at once whose kernels are the same
instantiation but ask for different amounts of shared memory: every call
succeeds and returns what it returns alone.  The most a launch may ask for is
an attribute of the kernel on its device, not of the call, so one call's
setting must not take away what another call's launch needs."""
import ctypes
import os
import subprocess

import pytest

from paper_2202_13951_gb300 import workloads
from test_gpu_parity import orbg  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CAP = 2000


@pytest.fixture(scope="module")
def native(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("threads") / "libthreads_host.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-pthread",
                           os.path.join(HERE, "threads_host.cpp"), "-o", out])
    return ctypes.CDLL(out)


class Call(ctypes.Structure):
    _fields_ = [("handle", ctypes.c_void_p), ("llr", ctypes.c_void_p),
                ("blocks", ctypes.c_int64), ("cw", ctypes.c_void_p), ("q", ctypes.c_void_p),
                ("ab", ctypes.c_void_p), ("stream", ctypes.c_void_p)]


def together(native, function, batched, jobs, calls):
    """jobs: (handle, code, blocks), one thread each."""
    threads = len(jobs)
    arr = (Call * threads)()
    bufs, streams = [], []
    for i, (handle, code, blocks) in enumerate(jobs):
        llr = torch.from_numpy(workloads.awgn_llr(code, blocks, 6.0, 92 + i)[0]).cuda()
        out = (torch.empty((blocks, code.n), dtype=torch.uint8, device="cuda"),
               torch.empty(blocks, dtype=torch.int32, device="cuda"),
               torch.empty(blocks, dtype=torch.uint8, device="cuda"))
        streams.append(torch.cuda.Stream())
        bufs.append((llr, out))
        arr[i] = Call(handle, llr.data_ptr(), blocks, *[t.data_ptr() for t in out],
                      streams[i].cuda_stream)
    refused = (ctypes.c_int * threads)()
    fn = ctypes.cast(function, ctypes.c_void_p)
    args = (None, fn) if batched else (fn, None)

    def outputs():
        torch.cuda.synchronize()
        got = [[t.clone() for t in out] for _, out in bufs]
        for _, out in bufs:
            for t in out:
                t.fill_(77)
        torch.cuda.synchronize()
        return got

    for i in range(threads):  # each alone
        native.calls_together(*args, ctypes.c_uint32(CAP), ctypes.byref(arr[i]), 1, 1,
                              ctypes.byref(refused, 4 * i))
    alone = outputs()
    assert list(refused) == [0] * threads
    native.calls_together(*args, ctypes.c_uint32(CAP), arr, threads, calls, refused)
    assert list(refused) == [0] * threads, "calls refused, of %d a thread" % calls
    for got, want in zip(outputs(), alone):
        for g, w in zip(got, want):
            assert torch.equal(g, w)


def test_plain_calls_of_different_lengths(orbg, native):  # noqa: F811
    codes = {n: workloads.rlc(n, n - 16, 91) for n in (200, 256)}
    handles = {n: orbg.Code(c.H, max_query_cap=CAP) for n, c in codes.items()}
    together(native, orbg.load_library().orbg_decode, False,
             [(handles[n].handle.value, codes[n], 16) for n in (256, 200, 256, 200)], 20000)


def test_batched_calls_of_different_sizes(orbg, native):  # noqa: F811
    """One set, batches that take eight and six warps a CTA."""
    code = workloads.rlc(256, 240, 91)
    handle = orbg.Code(code.H, max_query_cap=CAP)
    cs = orbg.CodeSet([handle])
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    together(native, orbg.load_library().orbg_decode_batched, True,
             [(cs.handle.value, code, 2 * sms * w) for w in (8, 6, 8, 6)], 5000)

"""The dispatch layer without a GPU: the memory it hands to the kernels, over the runtime of tests/host_runtime.cu."""
import ctypes
import os
import subprocess
import threading

import numpy as np
import pytest

from paper_2403_10444_b200 import build as bv_build

HERE = os.path.dirname(os.path.abspath(__file__))
F32, BF16 = 0, 1


@pytest.fixture(scope="module")
def host_so(tmp_path_factory):
    lib = bv_build.build()
    out = str(tmp_path_factory.mktemp("host") / "host_runtime.so")
    # (the plans are the library's own; names that both define bind to this file's)
    subprocess.check_call([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17",
                           "-Xcompiler", "-fPIC", "-shared", "-I", bv_build.CSRC, os.path.join(HERE, "host_runtime.cu"), "-o", out,
                           "-Xlinker", "-Bsymbolic", "-Xlinker", "-rpath=" + os.path.dirname(lib), lib])
    return ctypes.CDLL(out)


@pytest.fixture
def host(host_so):
    host_so.bv_release()
    host_so.host_errors.restype = ctypes.c_char_p
    host_so.host_live_bytes.restype = ctypes.c_size_t
    yield host_so
    host_so.bv_release()
    host_so.bv_set_option(b"kernel", 0)


FLOAT = ctypes.c_float(1.0)


def verify(host, B, gamma, V, dtype=BF16, fn="bv_verify", offset=0, diagnostics=False, stream=None):
    """One call on tensors that are never touched, `offset` elements off a 16-byte boundary; (status, kernel)."""
    p = ctypes.c_void_p
    base = (1 << 40) + offset * (4 if dtype == F32 else 2)
    x = p(1 << 41)
    args = [p(base), p(base + (1 << 39)), x, x]
    if "lse" in fn:
        args.append(x)
    args += [B, gamma, V, dtype]
    if "probs" not in fn:
        args.append(FLOAT)
    args += [x, x]
    if diagnostics:
        fn = fn if "probs" in fn else fn + "_ex"
        args += [x] * (3 if "probs" in fn else 5)
    elif "probs" in fn:
        args += [None] * 3
    status = getattr(host, fn)(*args, p(stream))
    return status, host.bv_last_kernel()


# batches that go through the phase kernel in parts, the last of which needs more scratch a sequence than the others
@pytest.mark.parametrize("B,gamma,V,dtype", [(1533, 2, 5089, BF16), (1533, 2, 2534, F32), (1533, 1, 10001, BF16), (1524, 1, 4601, BF16),
                                             (2000, 2, 1003, BF16), (769, 3, 50257, BF16)])
def test_every_part_of_a_batch_fits_the_workspace(host, B, gamma, V, dtype):
    for fn in ("bv_verify", "tv_verify"):
        host.bv_release()
        assert verify(host, B, gamma, V, dtype, fn) == (0, 5)
        assert host.host_errors() == b""


def test_scratch_fits_over_the_range(host):
    for B in (1, 3, 24, 33, 200, 700, 800, 1500, 1600):
        for gamma in (1, 2, 7, 33):
            for V in (1, 1003, 4096, 8209, 50257, 65536):
                for fn in ("bv_verify", "tv_verify", "bv_verify_lse", "bv_verify_probs"):
                    if V % 8 and ("lse" in fn or "probs" in fn):
                        continue
                    assert verify(host, B, gamma, V, fn=fn)[0] == 0
                    assert host.host_errors() == b"", (B, gamma, V, fn)


# calls of every kernel and of several sizes on one stream: (entry point, B, gamma, V, with diagnostics)
CALLS = [("bv_verify", 128, 8, 128256, False), ("bv_verify", 128, 8, 128256, True), ("bv_verify", 256, 8, 256000, False),
         ("tv_verify", 256, 8, 152064, False), ("bv_verify_lse", 256, 8, 152064, False), ("bv_verify", 4, 4, 32768, False),
         ("bv_verify", 700, 2, 5089, False), ("tv_verify", 24, 5, 50257, False), ("bv_verify", 2000, 16, 4096, False),
         ("bv_verify_probs", 400, 8, 152064, False), ("bv_verify", 100, 1, 1001, False)]


def call(host, c):
    assert verify(host, c[1], c[2], c[3], fn=c[0], diagnostics=c[4])[0] == 0
    return host.bv_last_kernel()


def test_the_calls_below_reach_every_kernel_that_keeps_scratch(host):
    assert {call(host, c) for c in CALLS} >= {1, 4, 5}


@pytest.mark.parametrize("warm", [True, False])
@pytest.mark.parametrize("a", CALLS)
def test_a_graph_replayed_between_eager_calls(host, a, warm):
    # whatever ran on the stream before or since, a replayed call finds its memory, zero where it has to be, and leaves the
    # eager calls' memory as they expect it
    for b in CALLS:
        host.bv_release()
        if warm:
            call(host, a)
        host.host_begin_capture(None)
        kernel = call(host, a)
        graph = host.host_end_capture()
        assert host.host_errors() == b"", (a, b)
        assert call(host, a) == kernel                    # captured or not: the same kernel
        for step in (b, graph, b, a, graph, graph, b):
            host.host_replay(graph) if step is graph else call(host, step)
            assert host.host_errors() == b"", (a, b)


def test_the_workspace_is_bounded_and_given_back(host):
    call(host, CALLS[0])
    for B in range(1, 600, 7):                            # grows many times
        call(host, ("bv_verify", B, 8, 128256, False))
    sizes = host.host_live_bytes()
    host.bv_release()
    for c in (("bv_verify", 595, 8, 128256, False), ("bv_verify", 130, 8, 128256, False)):
        call(host, c)
    assert sizes <= 5 * host.host_live_bytes()
    host.bv_release()
    assert host.host_live_bytes() == 0 and host.host_errors() == b""


@pytest.mark.parametrize("esz", [2, 4])
def test_a_vector_at_the_edge_of_a_tensor_of_any_size(host, esz):
    # the elements of a 16-byte vector that lie in a tensor, which may hold more of them than 32 bits count
    ull, first, n = ctypes.c_ulonglong, ctypes.c_int(), ctypes.c_int()
    for count in (1, 3, 7, 8, 9, 1000, 2 ** 31 - 1, 2 ** 31, 2 ** 31 + 5, 2 ** 32 + 1, 2 ** 33):
        for offset in range(0, 16, esz):
            lo = (1 << 40) + offset
            hi = lo + count * esz
            for p in {lo - offset, (hi - 1) // 16 * 16}:
                host.host_elements_inside(ull(p), ull(lo), ull(hi), esz, ctypes.byref(first), ctypes.byref(n))
                inside = [j for j in range(16 // esz) if lo <= p + j * esz < hi]
                assert list(range(first.value, n.value)) == inside, (count, offset, p)


def test_smoke_expects_the_kernels_that_run(host):
    import __graft_entry__ as entry
    for B, option, kernel in entry.SMOKE_CALLS:
        host.bv_set_option(b"kernel", option)
        for fn in ("bv_verify_ex", "tv_verify_ex", "gbv_verify_ex"):
            assert verify(host, B, 4, 32768, fn=fn[:-3], diagnostics=True) == (0, kernel), (B, option, fn)


def test_a_probe_of_the_decoding_loop_says_what_the_call_does_and_launches_nothing(host):
    for algo in (0, 1):
        for lse in (0, 1):
            for B, gamma, V in ((1, 1, 8), (3, 5, 4096), (33, 8, 16384), (768, 64, 32768), (769, 2, 4096), (32, 64, 65536), (3, 2, 8209), (2, 65, 4096)):
                before = host.host_launches()
                status = host.host_tables(algo, B, gamma, V, BF16, lse, 1)
                assert host.host_launches() == before and host.host_errors() == b""
                assert status == (-2 if B > 768 or V % 8 or gamma > 64 else 0)
                assert host.host_tables(algo, B, gamma, V, BF16, lse, 0) == status
                assert host.host_launches() == before + (status == 0)


def test_without_room_for_a_cooperative_launch_another_kernel_takes_the_call(host):
    # (a part of the GPU's SMs only, as under a percentage of its threads: the kernels that need one CTA on every SM are refused)
    host.host_refuse_cooperative(1)
    try:
        for fn in ("bv_verify", "tv_verify", "gbv_verify", "bv_verify_lse", "bv_verify_probs"):
            for B in (2, 12, 40, 800):
                for V in (4096, 128256) + ((50257,) if fn in ("bv_verify", "tv_verify") else ()):
                    assert verify(host, B, 5, V, fn=fn) == (0, 3 if V % 8 else 1), (fn, B, V)
        assert host.host_tables(1, 40, 5, 4096, BF16, 1, 0) == -2
        host.bv_set_option(b"kernel", 5)
        assert verify(host, 40, 5, 4096) == (0, 2)
    finally:
        host.host_refuse_cooperative(0)
    assert host.host_errors() == b"" and host.bv_last_cuda_error() == 0


# calls on both sides of the lines between the kernels: (entry point, B, gamma, V, dtype, diagnostics), kernel
ROUTES = [
    # rows that are not whole vectors: the element-wise kernel for a few short ones a sequence, if all sequences are at work at once
    (("tv_verify", 148, 5, 4099, BF16, False), 3), (("tv_verify", 148, 6, 4099, BF16, False), 5), (("tv_verify", 149, 5, 4099, BF16, False), 5),
    (("tv_verify", 148, 3, 8209, BF16, False), 3), (("tv_verify", 148, 4, 8209, BF16, False), 5), (("tv_verify", 148, 3, 8209, F32, False), 3),
    (("tv_verify", 148, 1, 16421, BF16, False), 5), (("tv_verify", 296, 1, 4099, BF16, False), 3), (("tv_verify", 297, 1, 4099, BF16, False), 5),
    (("tv_verify", 40, 2, 8209, F32, False), 3), (("tv_verify", 40, 3, 8209, F32, False), 5), (("tv_verify", 200, 2, 2051, BF16, False), 3),
    (("tv_verify", 200, 2, 4099, BF16, False), 5), (("tv_verify", 32, 2, 8209, F32, False), 3), (("tv_verify", 64, 1, 16421, BF16, False), 3), (("tv_verify", 33, 1, 32771, BF16, False), 5), (("tv_verify", 32, 2, 2051, BF16, False), 3),
    (("tv_verify", 32, 2, 4099, BF16, False), 4), (("tv_verify", 32, 2, 16421, BF16, False), 3), (("tv_verify", 16, 2, 16421, BF16, False), 4),
    (("bv_verify", 148, 2, 4099, BF16, False), 3), (("bv_verify", 148, 3, 4099, BF16, False), 5), (("bv_verify", 148, 3, 2051, BF16, False), 3),
    (("bv_verify", 148, 1, 8209, F32, False), 3), (("bv_verify", 148, 2, 8209, BF16, False), 5), (("bv_verify", 149, 1, 1003, BF16, False), 5),
    (("bv_verify", 32, 1, 1003, BF16, False), 4), (("bv_verify", 24, 5, 50257, BF16, False), 4), (("bv_verify", 150, 8, 50257, BF16, True), 5),
    # probabilities
    (("bv_verify_probs", 16, 4, 152064, BF16, False), 4), (("bv_verify_probs", 17, 4, 152064, BF16, False), 5), (("bv_verify_probs", 64, 8, 128256, BF16, False), 5),
    (("bv_verify_probs", 24, 16, 8192, BF16, False), 1), (("bv_verify_probs", 24, 13, 8192, BF16, False), 5), (("bv_verify_probs", 48, 16, 8192, BF16, False), 5),
    (("tv_verify_probs", 148, 8, 32768, BF16, False), 5), (("tv_verify_probs", 256, 8, 32768, BF16, False), 1), (("tv_verify_probs", 24, 8, 152064, F32, False), 1),
    (("bv_verify_probs", 100, 1, 152064, F32, False), 1), (("bv_verify_probs", 100, 1, 152064, BF16, False), 5),
    # every position swept
    (("bv_verify", 40, 8, 256000, BF16, True), 1), (("bv_verify", 40, 4, 256000, BF16, True), 5), (("bv_verify", 24, 16, 152064, BF16, True), 1),
    (("bv_verify", 64, 16, 65536, BF16, True), 5), (("bv_verify", 128, 8, 32768, F32, True), 1), (("bv_verify", 128, 4, 32768, F32, True), 5),
    (("bv_verify", 64, 12, 8192, F32, True), 5), (("bv_verify", 128, 12, 8192, F32, True), 1), (("bv_verify", 16, 8, 152064, BF16, True), 4),
    (("bv_verify", 32, 4, 152064, BF16, True), 5),
    # few sequences of long rows
    (("bv_verify_lse", 6, 8, 152064, F32, False), 4), (("bv_verify_lse", 10, 8, 152064, F32, False), 5), (("tv_verify_lse", 10, 8, 152064, F32, False), 4),
    (("tv_verify_lse", 10, 12, 152064, BF16, False), 5), (("bv_verify", 3, 16, 256000, F32, False), 1), (("bv_verify", 9, 16, 256000, F32, False), 1),
    (("bv_verify", 7, 16, 256000, BF16, False), 5), (("bv_verify", 7, 16, 128000, F32, False), 5),
    # the ordinary batches
    (("bv_verify", 1, 8, 152064, BF16, False), 4), (("bv_verify", 8, 8, 32000, F32, False), 4), (("bv_verify", 64, 8, 128256, BF16, False), 5),
    (("bv_verify", 96, 12, 152064, BF16, False), 5), (("bv_verify", 256, 8, 256000, BF16, False), 1), (("tv_verify", 256, 8, 152064, BF16, False), 1),
    (("bv_verify_lse", 64, 8, 128256, BF16, False), 5), (("gbv_verify", 64, 8, 128256, BF16, False), 5),
]


def test_which_kernel_takes_a_call(host):
    for (fn, B, gamma, V, dtype, diagnostics), kernel in ROUTES:
        assert verify(host, B, gamma, V, dtype, fn, diagnostics=diagnostics) == (0, kernel), (fn, B, gamma, V, dtype, diagnostics)
    assert host.host_errors() == b""


@pytest.mark.parametrize("devices,together", [((0, 1), 2), ((0, 0), 1)])
def test_host_buffers_are_shared_by_a_device_s_calls_and_by_no_others(host, devices, together):
    # two threads' calls of different sizes: on two devices both are under way at once, on one device one after the other
    status = []

    def call(device, B):
        host.host_set_device(device)
        gamma, V = 2, 64
        a = [np.zeros(n, np.float32) for n in (B * (gamma + 1) * V, B * gamma * V, B * gamma, B * (gamma + 2), B * (gamma + 1), B)]
        p = [ctypes.c_void_p(x.ctypes.data) for x in a]
        status.append(host.bv_verify_host(*p[:4], B, gamma, V, F32, FLOAT, *p[4:]))

    for d in set(devices):
        warm = threading.Thread(target=call, args=(d, 1))
        warm.start()
        warm.join()
    host.host_meet(2)
    try:
        threads = [threading.Thread(target=call, args=(d, B)) for d, B in zip(devices, (3, 40))]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    finally:
        met = host.host_met()
        host.host_meet(0)
    assert met == together and status == [0] * len(status) and host.host_errors() == b""
    for d in set(devices):
        release = threading.Thread(target=lambda: (host.host_set_device(d), host.bv_release()))
        release.start()
        release.join()


# (V, dtype, B, gamma, Algorithm 1), on both sides of the lines between the decoding loop in one kernel and in two launches an iteration
@pytest.mark.parametrize("call,one", [((16384, BF16, 128, 5, 0), 1), ((16384, BF16, 768, 32, 0), 1), ((16384, BF16, 8, 17, 0), 0), ((16384, BF16, 8, 24, 1), 1),
                                      ((16392, BF16, 8, 5, 0), 1), ((16392, BF16, 8, 6, 0), 0), ((16392, BF16, 8, 7, 1), 1), ((16392, BF16, 9, 6, 0), 1),
                                      ((2048, BF16, 148, 16, 0), 1), ((1024, BF16, 8, 64, 1), 1), ((1032, BF16, 8, 13, 0), 0), ((1024, F32, 8, 64, 0), 1), ((2048, BF16, 149, 16, 0), 0), ((2048, BF16, 592, 3, 0), 1), ((2048, BF16, 768, 4, 0), 0),
                                      ((32768, BF16, 148, 32, 0), 1), ((32768, BF16, 149, 6, 0), 0), ((32768, BF16, 445, 3, 0), 0), ((51200, BF16, 24, 4, 0), 0),
                                      ((51200, BF16, 25, 5, 0), 1), ((51200, BF16, 149, 3, 0), 0), ((51200, BF16, 593, 1, 0), 0), ((53256, BF16, 100, 1, 0), 0), ((8192, F32, 768, 64, 0), 1),
                                      ((24576, F32, 592, 3, 0), 1), ((24576, F32, 593, 3, 0), 0), ((26624, F32, 1, 2, 0), 1), ((26628, F32, 1, 1, 0), 0)])
def test_where_the_decoding_loop_is_one_kernel(host, call, one):
    assert host.host_loop_pays(*call) == one

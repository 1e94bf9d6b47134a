"""The library's host code over a stand-in for the CUDA runtime (fake_cudart.cpp): what it asks of streams and devices,
checked without a GPU."""
import concurrent.futures
import ctypes
import importlib.util
import os
import re
import subprocess

import numpy as np
import pytest

from paper_2609_22106_b200 import build, synth

HERE = os.path.dirname(os.path.abspath(__file__))
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


@pytest.fixture(scope="session")
def fake(tmp_path_factory):
    """The binding over a build of the library whose CUDA runtime is the stand-in."""
    d = tmp_path_factory.mktemp("fake_runtime")
    flags = ["-gencode", "arch=compute_100a,code=compute_100a", "-std=c++17", "-Xcompiler", "-fPIC", "-I", build.INCLUDE, "-I", build.CSRC]
    # (the stand-in first: its objects exist before the other files register their kernels)
    sources = [os.path.join(HERE, "fake_cudart.cpp")] + [os.path.join(build.CSRC, s) for s in build.SOURCES]
    objects = [str(d / (os.path.basename(s) + ".o")) for s in sources]
    with concurrent.futures.ThreadPoolExecutor(8) as pool:
        list(pool.map(lambda so: subprocess.check_call([NVCC, *flags, "-c", "-o", so[1], so[0]]), zip(sources, objects)))
    lib = str(d / "libprq_fake.so")
    subprocess.check_call(["g++", "-shared", "-Wl,-Bsymbolic", "-o", lib, *objects, "-lpthread"])
    spec = importlib.util.spec_from_file_location("prq_fake_binding", os.path.join(os.path.dirname(build.CSRC), "binding.py"))
    binding = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(binding)
    binding.LIB_PATH = lib
    binding.lib().fake_last_kernel.restype = ctypes.c_char_p
    return binding


def _device_weights(fake, N, K, k, experts=1):
    """A handle whose codes and scale bytes live on the device only."""
    W = np.stack([synth.weights(3 + e, N, K) for e in range(experts)])
    h = ctypes.c_void_p()
    amax = np.ones((experts, K), np.float32)
    fake._check(fake.lib().prq_prepare_weights_device(W.ctypes.data, experts, N, K, amax.ctypes.data, 0.5, k, None, None, ctypes.byref(h)), "prepare")
    return fake.Weights(h)


@pytest.mark.parametrize("form", ["clone", "offline_copy"])
@pytest.mark.parametrize("where", ["device", "host"])
def test_a_copy_of_a_handle_is_complete_when_the_call_returns(fake, form, where):
    """Everything in the copy is written before prq_weights_clone / prq_weights_offline_copy returns: prq_weights_get reads
    through a stream of its own, and the caller's next call may be on any stream."""
    N, K, k = 64, 512, 64
    w = _device_weights(fake, N, K, k) if where == "device" else fake.prepare_weights(synth.weights(5, N, K), np.ones(K, np.float32), 0.5, k)
    assert fake.lib().fake_pending() == 0
    c = getattr(w, form)()
    assert fake.lib().fake_pending() == 0
    assert np.array_equal(c.get(fake.FIELD_CODES), w.get(fake.FIELD_CODES))
    assert np.array_equal(c.get(fake.FIELD_SCALES), w.get(fake.FIELD_SCALES))
    c.free()
    w.free()


def _aligned(n_bytes):
    """Host bytes on a 256-byte boundary (device memory to the stand-in)."""
    a = np.zeros(n_bytes + 256, np.uint8)
    return a[-a.ctypes.data % 256:][:n_bytes]


def _every_kernel(fake):
    """Calls that between them launch every kernel with a shared-memory opt-in, on the current device."""
    L, p = fake.lib(), lambda a: a.ctypes.data
    for N, K, M in ((256, 512, 1), (256, 512, 32), (256, 512, 64), (256, 512, 128), (19456, 32, 64), (19456, 32, 128), (256, 512, 300),
                    (2560, 512, 2048), (2560, 512, 4096), (32, 9728, 2048)):
        w = fake.prepare_weights(np.zeros((N, K), np.uint16), np.ones(K, np.float32), 0.5, 0)
        x, codes, sf, y = (_aligned(n) for n in (M * K * 2, fake.act_bytes(M, K, 0, 1, fake.BUF_CODES), fake.act_bytes(M, K, 0, 1, fake.BUF_SCALES_SF), M * N * 4))
        ws = _aligned(max(16, fake.linear_workspace_bytes(w, M)))
        fake._check(L.prq_quantize_act(w.handle, fake.ACT_SCALE_PERM, p(x), M, K, None, p(codes), None, p(sf), None), f"quantize {N} {K} {M}")
        fake._check(L.prq_linear(w.handle, p(codes), p(sf), M, p(y), N, fake.F32, p(ws), ws.size, None), f"linear {N} {K} {M}")
        if M <= 128:
            two = (ctypes.c_void_p * 2)
            fake._check(L.prq_linear_multi(2, two(w.handle.value, w.handle.value), two(p(codes), p(codes)), two(p(sf), p(sf)), M, two(p(y), p(y)),
                                           (ctypes.c_int * 2)(N, N), fake.F32, None), f"multi {N} {K} {M}")
        if M <= fake.FUSED_MAX_M:
            fake._check(L.prq_linear_fused(w.handle, fake.ACT_IDENTITY, p(x), M, K, p(y), N, fake.F32, None), "fused")
        w.free()
    for N, M in ((128, 64), (1024, 1300), (2048, 1500), (6144, 700), (6144, 4096)):   # MXFP8: both kernels, several widths
        w = fake.prepare_weights(np.zeros((N, 256), np.uint16), np.ones(256, np.float32), 0.5, 0, fmt=fake.FMT_MXFP8)
        codes, sf, y = _aligned(M * 256), _aligned(L.prq_act_bytes_for(w.handle, M, fake.BUF_SCALES_SF)), _aligned(M * N * 4)
        fake._check(L.prq_linear(w.handle, p(codes), p(sf), M, p(y), N, fake.F32, None, 0, None), f"mxfp8 {N} {M}")
        w.free()
    E, N, K = 2, 512, 256   # stacked experts: quantiser, 64- and 128-token tiles, CTA pairs
    w = fake.prepare_weights(np.zeros((E, N, K), np.uint16), np.ones((E, K), np.float32), 0.5, 0)
    for M in (100, 300, 60000):
        codes, sf, x, y = _aligned(M * K // 2), _aligned(fake.act_bytes(M, K, 0, E, fake.BUF_SCALES_SF)), _aligned(M * K * 2), _aligned(M * N * 2)
        off = np.array([0, M // 2, M], np.int32)
        fake._check(L.prq_quantize_act(w.handle, fake.ACT_SCALE_PERM, p(x), M, K, p(off), p(codes), None, p(sf), None), f"grouped quantize {M}")
        fake._check(L.prq_linear_grouped(w.handle, p(codes), p(sf), p(off), M, p(y), N, fake.BF16, None), f"grouped {M}")
    w.free()
    gu = fake.prepare_weights(np.zeros((512, 256), np.uint16), np.ones(256, np.float32), 0.5, 0, gated_producer=True)
    down = fake.prepare_weights(np.zeros((64, 256), np.uint16), np.ones(256, np.float32), 0.5, 0)
    M = 300
    b = [_aligned(fake.act_bytes(M, 256, 0, 1, k)) for k in (fake.BUF_CODES, fake.BUF_SCALES_SF)]
    fake._check(L.prq_linear_gated(gu.handle, p(b[0]), p(b[1]), M, down.handle, p(b[0]), None, p(b[1]), None, None), "gated")
    gu.free()
    down.free()
    fake._check(L.prq_mxf4_peak_probe(4, None, None), "probe")


def test_every_kernel_runs_on_a_second_device(fake):
    """The shared-memory opt-in of a kernel belongs to a device: a process with handles on two GPUs needs it on both."""
    launches = []
    for device in (0, 1):
        assert fake.lib().cudaSetDevice(device) == 0
        try:
            before = fake.lib().fake_launches(device)
            _every_kernel(fake)
            launches.append(fake.lib().fake_launches(device) - before)
        finally:
            fake.lib().cudaSetDevice(0)
    assert launches[0] == launches[1]


def _quantise(fake, K, M, k=0, experts=1, layers=1):
    """One scale + permute launch; returns the kernel it took and its CTAs."""
    L, p = fake.lib(), lambda a: a.ctypes.data
    ws = [_device_weights(fake, 8, K, k, experts) for _ in range(layers)]
    x = _aligned(M * K * 2)
    codes, sf = _aligned(fake.act_bytes(M, K, k, experts, fake.BUF_CODES)), _aligned(fake.act_bytes(M, K, k, experts, fake.BUF_SCALES_SF))
    off = np.linspace(0, M, experts + 1).astype(np.int32)
    if layers == 1:
        fake._check(L.prq_quantize_act(ws[0].handle, fake.ACT_SCALE_PERM, p(x), M, K, p(off) if experts > 1 else None, p(codes), None, p(sf), None), "quantise")
    else:
        arr = ctypes.c_void_p * layers
        fake._check(L.prq_quantize_act_multi(layers, arr(*[w.handle.value for w in ws]), fake.ACT_SCALE_PERM, p(x), M, K, arr(*[p(codes)] * layers),
                                             arr(*[p(sf)] * layers), None), "quantise_multi")
    for w in ws:
        w.free()
    name = L.fake_last_kernel().decode()
    return "columns" if "quant_act_cols_kernel" in name else "atoms", L.fake_last_grid()


@pytest.mark.parametrize("K,layers,M,ctas", [
    (2560, 3, 1, 192), (2560, 3, 16, 192), (2560, 3, 64, 192), (2560, 4, 64, 256), (2560, 3, 96, 288),   # 3 x 128 of 444 places: fewer
    (2560, 2, 64, 256), (1024, 3, 64, 384)])                                                             # room enough: a row per CTA
def test_a_few_rows_for_several_layers_leave_room_for_the_next_launch(fake, K, layers, M, ctas):
    assert _quantise(fake, K, M, k=64, layers=layers) == ("columns", ctas)


@pytest.mark.parametrize("want,K,M,k,experts", [
    # rows of which two do not fit twice, up to the widest that one did
    ("columns", 25728, 300, 64, 1), ("atoms", 25760, 300, 64, 1), ("atoms", 28672, 4096, 64, 1), ("atoms", 51456, 16, 0, 1),
    # a CTA per SM from the atoms alone, two to 32 rows
    ("columns", 18816, 8, 64, 1), ("atoms", 18944, 8, 64, 1), ("columns", 18944, 1, 64, 1), ("atoms", 22016, 32, 0, 1), ("columns", 22016, 33, 64, 1),
    # nothing scattered to gather, 41 (65) to 128 rows of a narrow layer
    ("columns", 2560, 40, 0, 1), ("atoms", 2560, 41, 0, 1), ("atoms", 2560, 128, 0, 1), ("columns", 2560, 129, 0, 1), ("columns", 2560, 64, 32, 1),
    ("atoms", 2560, 65, 32, 1), ("columns", 2560, 65, 64, 1), ("columns", 1024, 64, 0, 1), ("atoms", 6144, 64, 0, 1), ("columns", 8192, 64, 0, 1),
    # stacked experts: one atom, a handful of atoms, a few rows, and what the structure is for
    ("atoms", 128, 2000, 32, 8), ("columns", 160, 9000, 32, 8), ("atoms", 256, 3800, 32, 2), ("columns", 256, 4000, 32, 2), ("atoms", 3072, 128, 64, 2),
    ("columns", 3072, 129, 64, 2), ("columns", 2048, 64, 64, 8), ("columns", 640, 128, 64, 16), ("atoms", 256, 128, 64, 32),
    ("columns", 384, 512, 64, 32), ("atoms", 384, 512, 64, 64), ("columns", 384, 2048, 64, 64), ("columns", 12864, 600, 64, 2), ("atoms", 12896, 600, 64, 2)])
def test_which_structure_quantises(fake, want, K, M, k, experts):
    assert _quantise(fake, K, M, k, experts)[0] == want


@pytest.mark.parametrize("want,E,N,K,M,bf16", [
    # the benchmark's expert projection at prefill; few tiles for the pairs; the padding of N; few tokens per expert
    ("pairs", 128, 2048, 768, 65536, True), ("tiles", 4, 1024, 256, 2048, True), ("tiles", 2, 1408, 768, 448, True), ("tiles", 128, 256, 768, 65536, True),
    ("pairs", 16, 1176, 352, 4688, True), ("tiles", 16, 600, 992, 3784, True), ("pairs", 128, 512, 768, 28672, True), ("tiles", 128, 512, 768, 28671, True),
    # long reductions: 512 tokens per expert and two tiles per pair
    ("pairs", 16, 1000, 2048, 8192, True), ("tiles", 16, 1000, 2048, 8191, True), ("tiles", 8, 1000, 2048, 5000, True), ("pairs", 128, 1408, 1280, 32768, True),
    ("tiles", 128, 1408, 1312, 32768, True),
    # fp32 output: long reductions and many tokens only
    ("tiles", 128, 2048, 768, 65536, False), ("pairs", 32, 2560, 1280, 24576, False), ("tiles", 32, 2560, 1280, 24575, False), ("tiles", 32, 2560, 1024, 24576, False)])
def test_which_tiles_the_grouped_product_takes(fake, want, E, N, K, M, bf16):
    W, amax, h = np.zeros((E, N, K), np.uint16), np.ones((E, K), np.float32), ctypes.c_void_p()
    fake._check(fake.lib().prq_prepare_weights_device(W.ctypes.data, E, N, K, amax.ctypes.data, 0.5, 0, None, None, ctypes.byref(h)), "prepare")
    w, off, some = fake.Weights(h), np.linspace(0, M, E + 1).astype(np.int32), _aligned(16)   # (nothing is read or written: the kernels do not run)
    fake._check(fake.lib().prq_linear_grouped(w.handle, some.ctypes.data, some.ctypes.data, off.ctypes.data, M, some.ctypes.data, (N + 7) // 8 * 8,
                                              fake.BF16 if bf16 else fake.F32, None), "grouped")
    assert ("pairs" if "grouped_pair" in fake.lib().fake_last_kernel().decode() else "tiles") == want
    w.free()


def test_a_workspace_of_its_own_belongs_to_the_stream_of_the_call(fake, monkeypatch):
    """linear() without a workspace on a stream that is not the current one: the workspace comes from that stream's memory
    pool and is cleared there, in front of the kernel that counts on it; it goes back to that pool when the call returns."""
    import contextlib

    import torch

    current, done = [None], []

    @contextlib.contextmanager
    def on(stream):
        current.append(stream)
        yield
        current.pop()

    class Side:
        cuda_stream = 0

    side, real_empty, real_zero = Side(), torch.empty, torch.Tensor.zero_
    monkeypatch.setattr(torch.cuda, "stream", on)
    monkeypatch.setattr(torch.cuda, "ExternalStream", lambda number, device: side)
    monkeypatch.setattr(torch, "empty", lambda *a, **k: (done.append(("empty", current[-1])), real_empty(*a, **k))[1])
    monkeypatch.setattr(torch.Tensor, "zero_", lambda t: (done.append(("zero", current[-1])), real_zero(t))[1])
    N, K, M = 256, 9728, 200        # a call that cuts its tiles along K
    w = fake.prepare_weights(np.zeros((N, K), np.uint16), np.ones(K, np.float32), 0.5, 0)
    t = lambda n: torch.frombuffer(memoryview(_aligned(n)), dtype=torch.uint8)
    codes, sf, y = t(M * K // 2), t(fake.act_bytes(M, K, 0, 1, fake.BUF_SCALES_SF)), t(M * N * 4).view(torch.float32).view(M, N)
    fake.linear(w, codes, sf, M, out=y, stream=side)
    assert done == [("empty", side), ("zero", side)]
    monkeypatch.undo()
    w.free()


def test_freeing_nothing_frees_nothing(fake):
    """prq_weights_free(NULL) is a no-op, also where the library itself calls it (the search's first candidate): what freed
    layers left to the next ones stays; prq_release_cached_memory gives it back."""
    L, K, k = fake.lib(), 512, 64
    fake.release_cached_memory()
    _device_weights(fake, 640, K, k).free()
    frees = L.fake_frees()
    L.prq_weights_free(None)
    assert L.fake_frees() == frees
    w, _, _ = fake.prepare_weights_search(synth.weights(3, 64, K), np.ones((8, K), np.uint16), [0.25, 0.5], k)
    mallocs = L.fake_mallocs()
    _device_weights(fake, 640, K, k).free()
    assert L.fake_mallocs() == mallocs       # the block of the first layer of this size was still there
    w.free()
    frees = L.fake_frees()
    fake.release_cached_memory()
    assert L.fake_frees() == frees + 3       # that layer's, and both candidates'


@pytest.mark.parametrize("what", ["host", "mxfp8", "device", "search", "clone", "offline_copy"])
def test_an_allocation_that_fails_is_tried_again_without_what_is_kept(fake, what):
    """Memory of freed layers goes back to the device before any allocation of the library gives up -- whichever it is."""
    L, N, K, k = fake.lib(), 64, 512, 64
    W, amax = synth.weights(3, N, K), np.ones(K, np.float32)
    original = _device_weights(fake, N, K, k)
    call = {"host": lambda: fake.prepare_weights(W, amax, 0.5, k), "mxfp8": lambda: fake.prepare_weights(W, amax, 0.5, 0, fmt=fake.FMT_MXFP8),
            "device": lambda: _device_weights(fake, N, K, k), "search": lambda: fake.prepare_weights_search(W, np.ones((200, K), np.uint16), [0.25, 0.5], k)[0],
            "clone": original.clone, "offline_copy": original.offline_copy}[what]
    nth = 1
    while True:
        fake.release_cached_memory()
        _device_weights(fake, 640, K, k).free()         # a block is kept, too large for anything in the call
        mallocs = L.fake_mallocs()
        L.fake_fail_malloc(nth)
        w = call()
        done = L.fake_mallocs() - mallocs < nth         # there was no nth allocation to fail
        L.fake_fail_malloc(0)
        w.free()
        if done:
            break
        mallocs = L.fake_mallocs()
        _device_weights(fake, 640, K, k).free()
        assert L.fake_mallocs() == mallocs + 1          # that block went back
        nth += 1
    assert nth > 1
    original.free()
    fake.release_cached_memory()


def _asks(fake, ws, M, mode):
    """One quantiser launch for the layers `ws`: what its instance asks for in L2 (its last template argument)."""
    L, p, K, n = fake.lib(), lambda a: a.ctypes.data, ws[0].K, len(ws)
    some, arr = _aligned(16), ctypes.c_void_p * n    # (nothing is read or written: the kernels do not run)
    if n == 1:
        fake._check(L.prq_quantize_act(ws[0].handle, mode, p(some), M, K, None, p(some), None, p(some), None), "quantise")
    else:
        fake._check(L.prq_quantize_act_multi(n, arr(*[w.handle.value for w in ws]), mode, p(some), M, K, arr(*[p(some)] * n), arr(*[p(some)] * n), None), "multi")
    cols, atoms = (re.search(rf"quant_act{kind}_kernelI\w*?L[bi](\d)EE", L.fake_last_kernel().decode()) for kind in ("_cols", ""))
    return ("nothing", "weights")[int(cols[1])] if cols else ("nothing", "rows", "weights")[int(atoms[1])]


@pytest.mark.parametrize("weights,Ns,K,M,gated", [
    (True, [2560], 4096, 1, False), (True, [2560], 4096, 128, False), (False, [2560], 4096, 129, False), (False, [2560], 4096, 2048, False),
    (False, [256], 256, 16, False), (False, [1024], 2560, 64, False), (True, [2560], 4064, 64, False), (False, [2560], 4064, 32, False), (False, [2560], 3264, 64, False), (True, [2560], 4128, 32, False), (True, [10240], 4096, 64, False),
    (False, [10240], 4128, 64, False), (True, [4096, 1024, 1024], 2560, 96, False), (False, [4096, 1024, 1024], 2560, 97, False), (False, [512, 256], 1024, 64, False),
    (False, [9728, 9728], 2560, 64, False), (False, [2560], 4096, 64, True)])
def test_what_a_quantiser_asks_for(fake, weights, Ns, K, M, gated):
    """5 (from 33 rows on: 4) to 20 MB of weights on up to 128 rows, not those of a gated producer; everything else takes the instances without hints, whose
    launches carry no parameters for them."""
    for mode, otherwise in ((fake.ACT_IDENTITY, "rows"), (fake.ACT_SCALE_PERM, "nothing")):
        ws = [_zero_weights(fake, N, K, gated=gated) for N in Ns]
        assert _asks(fake, ws, M, mode) == ("weights" if weights else otherwise), mode
        for w in ws:
            w.free()


@pytest.mark.parametrize("several", [False, True])
def test_a_quantiser_without_a_product_behind_it_asks_once(fake, several):
    """... and again once a product has been called, in whichever form."""
    ws = [_zero_weights(fake, N, 2560) for N in ((4096, 1024) if several else (4096,))]
    asked = lambda mode=fake.ACT_SCALE_PERM: _asks(fake, ws, 16, mode)
    products = [lambda: _cluster(fake, ws, 16)] + ([] if several else [lambda: _cluster(fake, ws, 16, fused=True)])
    for product in products:
        assert asked() == "weights"
        assert asked() == "nothing" and asked(fake.ACT_IDENTITY) == "nothing"
        product()
        assert asked() == "weights"
        product()
        product()
    if several:   # a product with one of the layers is not one with the other
        assert asked() == "weights"
        _cluster(fake, ws[:1], 16)
        assert asked() == "nothing"
    for w in ws:
        w.free()


def _zero_weights(fake, N, K, k=0, gated=False, stream=None):
    W, amax, h = np.zeros((N, K), np.uint16), np.ones(K, np.float32), ctypes.c_void_p()
    o = fake._opts(False, gated)
    fake._check(fake.lib().prq_prepare_weights_device(W.ctypes.data, 1, N, K, amax.ctypes.data, 0.5, k, ctypes.cast(ctypes.pointer(o), ctypes.c_void_p), stream,
                                                      ctypes.byref(h)), "prepare")
    return fake.Weights(h)


def _cluster(fake, ws, M, fused=False):
    """Cluster size of one decode launch over the layers `ws`."""
    L, p, n = fake.lib(), lambda a: a.ctypes.data, len(ws)
    some, arr = _aligned(16), ctypes.c_void_p * n    # (nothing is read or written: the kernels do not run)
    if fused:
        fake._check(L.prq_linear_fused(ws[0].handle, fake.ACT_IDENTITY, p(some), M, ws[0].K, p(some), ws[0].N, fake.F32, None), "fused")
    elif n == 1:
        fake._check(L.prq_linear(ws[0].handle, p(some), p(some), M, p(some), ws[0].N, fake.F32, None, 0, None), "linear")
    else:
        fake._check(L.prq_linear_multi(n, arr(*[w.handle.value for w in ws]), arr(*[p(some)] * n), arr(*[p(some)] * n), M, arr(*[p(some)] * n),
                                       (ctypes.c_int * n)(*[w.N for w in ws]), fake.F32, None), "multi")
    return L.fake_last_cluster()


@pytest.mark.parametrize("want,Ns,K,k,M", [
    (4, [4096], 2560, 128, 1), (4, [4096], 2560, 128, 16), (6, [2560], 4096, 256, 1), (8, [2560], 9728, 256, 16), (2, [9728], 2560, 256, 1),
    (3, [9728], 2560, 256, 32), (1, [12288], 1024, 0, 32), (8, [2560], 9728, 256, 17), (1, [19456], 1024, 0, 32), (1, [256], 128, 0, 4),
    # a quantiser in front of several layers
    (4, [2560, 2560], 4096, 128, 1), (5, [2560, 2560], 4096, 128, 32), (3, [4096, 1024, 1024], 2560, 128, 16), (2, [4096, 4096], 1024, 64, 16),
    # a CTA per SM
    (2, [4096, 1024, 1024], 2560, 128, 64), (2, [256], 256, 32, 128), (8, [512], 2560, 0, 64)])
def test_which_cluster_size_a_decode_call_takes(fake, want, Ns, K, k, M):
    ws = [_zero_weights(fake, N, K, k) for N in Ns]
    assert _cluster(fake, ws, M) == want
    for w in ws:
        w.free()


@pytest.mark.parametrize("form", ["device", "host", "clone", "offline_copy"])
@pytest.mark.parametrize("N,K,k", [(256, 256, 32), (2560, 4096, 256), (4096, 2560, 0), (5120, 512, 0)])
def test_one_launch_and_two_split_alike(fake, form, N, K, k):
    """prq_linear_fused gives the bits of the two calls: the same cluster size at every token count, whatever the handle's
    origin."""
    w = fake.prepare_weights(np.zeros((N, K), np.uint16), np.ones(K, np.float32), 0.5, k) if form == "host" else _zero_weights(fake, N, K, k)
    c = getattr(w, form)() if form in ("clone", "offline_copy") else w
    for M in range(1, fake.FUSED_MAX_M + 1):
        assert _cluster(fake, [c], M) == _cluster(fake, [c], M, fused=True) == _cluster(fake, [w], M), M
    for h in {c, w}:
        h.free()


@pytest.fixture
def empty_pool(fake):
    fake.release_cached_memory()
    yield fake.lib()
    fake.release_cached_memory()


def _allocates(fake, *a, **k):
    """Whether preparing the layer on the device allocates; frees it again."""
    before = fake.lib().fake_mallocs()
    _zero_weights(fake, *a, **k).free()
    return fake.lib().fake_mallocs() > before


def test_a_freed_layers_memory_serves_the_next_one_of_about_its_size(fake, empty_pool):
    assert _allocates(fake, 6400, 512)
    assert not _allocates(fake, 6400, 512) and not _allocates(fake, 5120, 512)    # all of the block, four fifths of it
    assert _allocates(fake, 4160, 512) and _allocates(fake, 12800, 512)           # two thirds, twice as much
    assert not any(_allocates(fake, N, 512) for N in (4160, 6400, 12800))         # the smallest that is large enough
    assert empty_pool.cudaSetDevice(1) == 0
    try:
        assert _allocates(fake, 6400, 512)                                        # another device's memory
    finally:
        empty_pool.cudaSetDevice(0)


def test_what_freed_layers_leave_is_bounded(fake, empty_pool):
    sizes = (64, 320, 1600, 8000, 40000)                       # none serves another one
    for N in sizes:
        assert _allocates(fake, N, 128)
    frees = empty_pool.fake_frees()
    assert not any(_allocates(fake, N, 128) for N in sizes[1:]) and _allocates(fake, sizes[0], 128)   # four blocks, the oldest went
    assert empty_pool.fake_frees() == frees + 1                # ... and the next oldest for it
    fake.release_cached_memory()
    assert _allocates(fake, 8192, 9728) and _allocates(fake, 13312, 9728)   # 52 and 84 MB: the first one makes room
    assert _allocates(fake, 8192, 9728)
    assert _allocates(fake, 17408, 9728) and _allocates(fake, 17408, 9728)  # 106 MB: never kept
    assert not _allocates(fake, 8192, 9728)


def _side_uses(fake):
    """Every call that queues work on a layer's memory, as (handles, call on a stream)."""
    L, p, some = fake.lib(), lambda a: a.ctypes.data, _aligned(1 << 16)
    two, ints = ctypes.c_void_p * 2, ctypes.c_int * 2
    one = lambda **k: [_zero_weights(fake, 256, 256, **k)]
    pair = lambda: [_zero_weights(fake, 256, 256) for _ in range(2)]
    hs = lambda ws: two(*[w.handle.value for w in ws])
    x = p(some)
    down = fake.prepare_weights(np.zeros((64, 256), np.uint16), np.ones(256, np.float32), 0.5, 0)   # (memory of its own)
    return {
        "quantize": (one, lambda ws, s: L.prq_quantize_act(ws[0].handle, 1, x, 4, 256, None, x, None, x, s)),
        "quantize_multi": (pair, lambda ws, s: L.prq_quantize_act_multi(2, hs(ws), 1, x, 4, 256, two(x, x), two(x, x), s)),
        "linear": (one, lambda ws, s: L.prq_linear(ws[0].handle, x, x, 4, x, 256, 0, None, 0, s)),
        "linear_multi": (pair, lambda ws, s: L.prq_linear_multi(2, hs(ws), two(x, x), two(x, x), 4, two(x, x), ints(256, 256), 0, s)),
        "fused": (one, lambda ws, s: L.prq_linear_fused(ws[0].handle, 0, x, 4, 256, x, 256, 0, s)),
        "grouped": (one, lambda ws, s: L.prq_linear_grouped(ws[0].handle, x, x, x, 4, x, 256, 0, s)),
        "static_scratch": (one, lambda ws, s: L.prq_linear_static_scratch(ws[0].handle, x, x, 200, x, 256, 0, s)),
        "gated": (lambda: [_zero_weights(fake, 512, 256, gated=True)],
                  lambda ws, s: L.prq_linear_gated(ws[0].handle, x, x, 4, down.handle, x, None, x, None, s)),
    }


@pytest.mark.parametrize("use", ["quantize", "quantize_multi", "linear", "linear_multi", "fused", "grouped", "static_scratch", "gated", "prepare"])
def test_memory_that_another_stream_may_read_is_not_kept(fake, empty_pool, use):
    """A layer that was prepared or used on any stream but the legacy one goes back to the device when it is freed -- its memory is
    not handed to a preparation that other stream's work is not ordered with -- and no preparation there gets kept memory."""
    L, stream = empty_pool, ctypes.c_void_p()
    assert L.cudaStreamCreateWithFlags(ctypes.byref(stream), 1) == 0
    try:
        if use == "prepare":
            assert _allocates(fake, 256, 256) and not _allocates(fake, 256, 256)   # a block is kept
            frees = L.fake_frees()
            assert _allocates(fake, 256, 256, stream=stream)
            assert L.fake_frees() == frees + 1
            return
        make, call = _side_uses(fake)[use]
        for s, kept in ((None, True), (stream, False)):
            fake.release_cached_memory()
            ws = make()
            assert call(ws, s) == 0
            frees = L.fake_frees()
            for w in ws:
                w.free()
            assert L.fake_frees() == frees + (0 if kept else len(ws)), s
    finally:
        L.cudaStreamDestroy(stream)

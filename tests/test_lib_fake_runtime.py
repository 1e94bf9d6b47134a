"""The library's host code over a stand-in for the CUDA runtime (fake_cudart.cpp): what it asks of streams and devices,
checked without a GPU."""
import concurrent.futures
import ctypes
import importlib.util
import os
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
    binding.lib()
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

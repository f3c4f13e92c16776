"""Contexts on several devices of one process: whether the level kernels may run in clusters of sixteen CTAs is decided,
and allowed, for every device by itself.  No GPU: the compiled k_node.cu is linked against a stand-in for the runtime
calls it makes (tests/fake_cudart.c), which keeps function attributes per device and refuses what the runtime refuses."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))

pytestmark = pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"),
                                reason="nvcc not available to build the library")


@pytest.fixture(scope="module")
def node(tmp_path_factory):
    from paper_2006_06537_gb300 import build

    build.build()
    obj = os.path.join(build.OUT, "k_node.o")
    if not os.path.exists(obj):
        build.build(force=True)
    d = tmp_path_factory.mktemp("node")
    so = str(d / "node.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run(["gcc", "-O1", "-I", inc, "-fPIC", "-c", os.path.join(HERE, "fake_cudart.c"),
                    "-o", str(d / "fake.o")], check=True)
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", so, obj, str(d / "fake.o")], check=True)
    return C.CDLL(so)


def _launch(node, ctas):
    """One node of rank <= 16 by a cluster of `ctas` (launch_node, C++ linkage)."""
    p, i, z = C.c_void_p(), C.c_int, C.c_size_t(0)
    fn = node["_Z11launch_nodePK8FactDesciibiiiPdPjPiiP11CUstream_stim"]
    return fn(p, i(16), i(-1), C.c_bool(True), i(0), i(1), i(ctas), p, p, p, i(-1), p, i(1), z)


def test_every_device_has_its_own_answer(node):
    largest = node["_Z16node_cluster_maxv"]
    for dev, holds in ((0, 1), (1, 1), (2, 0), (0, 1), (3, 1), (2, 0)):
        node.fake_device(dev, holds)
        c = largest()
        assert c == (16 if holds else 8), dev
        assert _launch(node, c) == 0, dev
        assert node.fake_last_cluster() == c

"""What the host side launches and on which device, with a stand-in for the CUDA
runtime (tests/fake_runtime.cpp) linked to the library's own objects: no GPU needed."""
import ctypes
import importlib.util
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    spec = importlib.util.spec_from_file_location("kcl_build", os.path.join(ROOT, "paper_2203_13512_gb300", "build.py"))
    b = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(b)
    b.build()
    objs = []
    for src in ("kcl_prep.cu", "kcl_sub.cu"):
        obj = os.path.join(b.BUILD, src + ".o")
        objs.append(obj if os.path.exists(obj) else b._compile(os.path.join(b.CSRC, src)))
    tmp = tmp_path_factory.mktemp("fake")
    objs.append(str(tmp / "probe.o"))
    subprocess.run([b.nvcc_path(), *b._flags(), "-c", os.path.join(ROOT, "tests", "launch_sub_probe.cu"), "-o",
                    objs[-1]], check=True)
    lib = str(tmp / "libfake.so")
    # symbols bound inside: the process may have the real runtime loaded as well
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic",
                    "-I" + os.path.join(os.path.dirname(os.path.dirname(b.nvcc_path())), "include"),
                    os.path.join(ROOT, "tests", "fake_runtime.cpp"), *objs, "-o", lib], check=True)
    lib = ctypes.CDLL(lib)
    lib.fake_launches.restype = ctypes.c_char_p

    def launches():
        """(device, kernel, blocks, threads, cluster) of the launches since the last look."""
        out = []
        for line in lib.fake_launches().decode().splitlines():
            dev, name, *rest = line.split()
            kernel = next((k for k in ("k_peel_grid", "k_peel_cluster", "k_peel_block", "k_sub_cta", "k_sub_warp")
                           if k in name), name)
            out.append((int(dev), kernel, *map(int, rest)))
        return out

    return lib, launches


def _order(lib, n):
    p = ctypes.cast(ctypes.create_string_buffer(64), ctypes.c_void_p)
    return lib.kcl_degeneracy_order_noalloc(ctypes.c_uint32(n), p, p, p, p, p, None)


def test_peel_cluster_on_every_device(fake):
    """The 16-CTA cluster needs an attribute that belongs to one device: a second
    device gets it too, whichever came first."""
    lib, launches = fake
    for dev in (3, 0, 3, 5):
        lib.fake_device(dev)
        assert _order(lib, 300_000) == 0
        got = launches()
        assert [(d, k) for d, k, *_ in got] == [(dev, "k_peel_grid"), (dev, "k_peel_cluster")]
        assert got[1][2] == got[1][4] == 16
        assert _order(lib, 20_000) == 0
        assert [(d, k, b) for d, k, b, *_ in launches()] == [(dev, "k_peel_cluster", 16)]
    lib.fake_device(0)


@pytest.mark.parametrize("k,c,listing", [(5, 4, 0), (6, 5, 0), (6, 1, 0), (4, 3, 1), (5, 2, 1), (6, 5, 1)])
def test_one_warp_per_root_has_no_shares(fake, k, c, listing):
    """A class of few roots: its roots are shared by several CTAs each, except when
    one warp is to walk a root's whole subtree (NodeParallel)."""
    lib, launches = fake
    assert lib.probe_launch_sub(k, c, 10, 1024, listing, 0) == 1
    (_, kernel, blocks, _, _), = launches()
    assert kernel == "k_sub_cta" and 10 < blocks <= 80
    assert lib.probe_launch_sub(k, c, 10, 1024, listing, 1) == 1
    (_, kernel, blocks, _, _), = launches()
    assert kernel == "k_sub_cta" and blocks == 10

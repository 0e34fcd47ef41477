"""Host code of the library on a fake CUDA runtime (tests/native): what its
launches, its server and its locks do when calls run side by side or fail.
The objects are the library's own; only the kernels' launches are stood in."""
import os
import subprocess

import pytest

import paper_2602_10080_gb300.buildlib as buildlib

HERE = os.path.dirname(os.path.abspath(__file__))
NATIVE = os.path.join(HERE, "native")
KERNELS = ["kernels_u32.o", "kernels_u32x.o", "kernels_f32.o", "kernels_f32x.o", "wave_kernels.o", "fan_kernels.o"]
HOST = ["sssp_api.o", "sssp_autotune.o", "sssp_serve.o", "sssp_noalloc.o", "sssp_wave.o", "sssp_layout.o"]


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    buildlib.build(force=not all(os.path.exists(os.path.join(buildlib.OBJ, o)) for o in KERNELS + HOST))
    out = tmp_path_factory.mktemp("native")
    cuda = os.path.dirname(os.path.dirname(buildlib._nvcc()))
    if not os.path.isdir(os.path.join(cuda, "include")):
        cuda = "/usr/local/cuda"
    fake = str(out / "fake_cuda.o")
    subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", f"-I{cuda}/include", "-c", os.path.join(NATIVE, "fake_cuda.cpp"),
                    "-o", fake], check=True)
    built = {}

    def go(name, objs, *args):
        if name not in built:
            exe = str(out / name)
            cmd = [buildlib._nvcc(), *buildlib.ARCH, "-O1", "-std=c++17", "-cudart", "shared", "-I", buildlib.CSRC,
                   "-I", NATIVE, os.path.join(NATIVE, name + ".cu"), fake,
                   *[os.path.join(buildlib.OBJ, o) for o in objs], "-o", exe, "-lpthread",
                   f"-Xlinker=-rpath={cuda}/lib64"]
            r = subprocess.run(cmd, capture_output=True, text=True)
            assert r.returncode == 0, r.stderr
            built[name] = exe
        r = subprocess.run([built[name], *args], capture_output=True, text=True, timeout=120)
        assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr

    return go


def test_shared_memory_limits_do_not_shrink(run):
    run("host_launch", KERNELS)


@pytest.mark.parametrize("what", ["destroyed", "turns", "places", "busy_stream", "no_memory", "smaller_jobs", "refused_launches",
                                  "fault", "time_limit", "autotune",
                                  "noalloc_without_clusters", "wide_fronts"])
def test_server(run, what):
    run("host_serve", HOST, what)

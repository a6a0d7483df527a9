"""Which kernels a step of fp32 precision takes where its stream has fewer SMs than a whole B200 (a partition, a context with
a share of the SMs): kernels whose blocks wait for one another need all of them resident at once, and the CUDA runtime refuses a launch
that is too large.  The library runs on a stand-in for the runtime (fewer_sms.c), without a GPU."""
import os
import re
import subprocess

import pytest

from paper_2410_01623_b200 import build as fbuild

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    lib = fbuild.build()
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    out = str(tmp_path_factory.mktemp("fewer_sms") / "fewer_sms")
    subprocess.run(["gcc", "-O1", "-o", out, os.path.join(HERE, "fewer_sms.c"), "-rdynamic", "-I", os.path.join(ROOT, "include"), "-I", cuda,
                    lib, "-Wl,-rpath," + os.path.dirname(lib), "-Wl,--unresolved-symbols=ignore-in-shared-libs"], check=True)
    return out


SEVERAL = ["k_back_project", "k_finalize", "k_back_project"]
LONG = ["k_split_projection", "k_part_project", "k_moments"]


@pytest.mark.parametrize("sms,share,call,matrix,count,kernels", [
    (148, 0, "list", (1280, 1280, 64), 1, ["k_project", "k_back_step<128>:101"]),
    (101, 0, "list", (1280, 1280, 64), 1, ["k_project", "k_back_step<128>:101"]),
    (100, 0, "list", (1280, 1280, 64), 1, ["k_project"] + SEVERAL),
    (148, 100, "list", (1280, 1280, 64), 1, ["k_project"] + SEVERAL),
    (89, 0, "list", (512, 1376, 128), 1, ["k_project", "k_back_step<64>:89"]),
    (88, 0, "list", (512, 1376, 128), 1, ["k_project", "k_back_step<128>:45"]),
    (148, 0, "single", (1280, 1280, 64), 1, ["k_noalloc_setup", "k_project", "k_back_step<128>:101"]),
    (100, 0, "single", (1280, 1280, 64), 1, ["k_noalloc_setup", "k_project"] + SEVERAL + ["k_noalloc_store_scalars"]),
    (148, 40, "single", (512, 1376, 128), 1, ["k_noalloc_setup", "k_project"] + SEVERAL + ["k_noalloc_store_scalars"]),
    (60, 0, "list", (512, 1376, 128), 56, LONG + ["k_part_step:60"]),
    (148, 60, "list", (512, 1376, 128), 56, LONG + ["k_part_step:60"]),
    (148, 40, "list", (1280, 1280, 128), 4, LONG + ["k_part_back", "k_finalize", "k_form_x", "k_part_back"]),
])
def test_kernels_of_a_step(program, sms, share, call, matrix, count, kernels):
    out = subprocess.run([program, str(sms), str(share), call, *map(str, matrix), str(count)], capture_output=True, text=True, timeout=60, check=True)
    launches, status = out.stdout.strip("\n").split("\n")[-2:]
    assert status.split()[0] == "0", status
    got = re.findall(r"\d(k_[a-z_]+?)(?:ILi(\d+)E\w*)?E[A-Zi]\w*:(\d+)", launches)
    assert len(got) == len(kernels), launches
    for (name, size, blocks), want in zip(got, kernels):
        if ":" in want:
            name += ("<%s>" % size if "<" in want else "") + ":" + blocks
        assert name == want, launches

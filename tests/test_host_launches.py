"""What the library's host code asks of the CUDA runtime, seen through a stand-in for it (fake_cuda_runtime.cpp; no GPU, no
device code runs): the launches of a call, and what a call does when one of them is refused."""
import json
import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2407_12077_b200", "csrc")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
pytestmark = pytest.mark.skipif(not os.path.exists(NVCC), reason="no nvcc")

# std::random_device may throw where the system has no source of random numbers
PRELUDE = """
#include <random>
#include <stdexcept>
namespace std { struct gf_refusing_device { unsigned operator()() { throw std::runtime_error("no random device"); } }; }
#define random_device gf_refusing_device
"""

CALLER = """
import ctypes, json, sys
lib = ctypes.CDLL(sys.argv[1])
lib.fake_log.restype = ctypes.c_char_p
P = lambda i: ctypes.c_void_p(0x10000000 * (i + 1))      # never dereferenced
WS = 0x700000000000
out = []
for name, args, refuse in json.loads(sys.stdin.read()):
    lib.fake_reset(*refuse)
    conv = []
    for i, a in enumerate(args):
        conv.append(P(i) if a == "p" else ctypes.c_void_p(WS) if a == "ws" else ctypes.c_size_t(a[0]) if isinstance(a, list) else
                    ctypes.c_longlong(a["ll"]) if isinstance(a, dict) else a if a is None else ctypes.c_int(a))
    status = getattr(lib, name)(*conv)
    out.append([status, lib.fake_log().decode().splitlines()])
print(json.dumps(out))
"""


@pytest.fixture(scope="module")
def host_library(tmp_path_factory):
    d = tmp_path_factory.mktemp("host")
    prelude, lib = str(d / "prelude.h"), str(d / "libhost.so")
    with open(prelude, "w") as f:
        f.write(PRELUDE)
    subprocess.run(["g++", "-shared", "-fPIC", "-I/usr/local/cuda/include", "-o", str(d / "libfake.so"),
                    os.path.join(ROOT, "tests", "fake_cuda_runtime.cpp")], check=True)
    subprocess.run([NVCC, "-gencode", "arch=compute_100a,code=compute_100a", "-std=c++17", "--expt-relaxed-constexpr", "-w",
                    "-include", prelude, "-Xcompiler", "-fPIC", "-shared", "-cudart", "none", "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", lib,
                    os.path.join(CSRC, "gf_wkv6_api.cu"), "-L", str(d), "-lfake", "-Xlinker", "-rpath", "-Xlinker", str(d)], check=True)
    return lib


def calls(lib, *todo):
    """[(status, log lines)] of the calls, made one after another in a process of their own."""
    r = subprocess.run([sys.executable, "-c", CALLER, lib], input=json.dumps(todo), capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr[-500:]
    return json.loads(r.stdout)


def backward(c2, B, T, H, bytes_):
    ins = ["p"] * 4 + ([] if c2 else ["p"]) + ["p"] * 3 + ["p"] * 4 + ([] if c2 else ["p"]) + ["p"]
    return ["gf_wkv6_backward" + ("_c2" if c2 else "") + "_saved", ins + [B, T, H, 64, "ws", [bytes_], None]]


@pytest.mark.parametrize("c2", [False, True])
def test_gradient_clears_the_words_of_its_cuts(host_library, c2):
    # a replayed graph repeats the call's launches with the arguments of the first time: the words that announce the adjoint at
    # a cut have to be cleared by the call itself, every time, before the launch that waits for them
    for s, log in calls(host_library, backward(c2, 5, 700, 32, 1 << 40) + [[0, 0]], backward(c2, 5, 700, 32, 1 << 40) + [[0, 0]]):
        assert s == 0
        cut = [i for i, line in enumerate(log) if " cooperative " in line]
        assert len(cut) == 1 and log[cut[0]].startswith("grid 148 "), log
        cleared = [line.split() for line in log[:cut[0]] if line.startswith("memset")]
        assert len(cleared) == 1 and cleared[0][2:] == ["0", str(8 * 148)], log
        assert int(cleared[0][1]) > 0x700000000000          # (in the workspace, behind the checkpoints)


@pytest.mark.parametrize("H,streamed", [(65536, True), (65537, False)])
def test_streams_end_where_a_head_no_longer_fits_its_descriptor(host_library, H, streamed):
    (s, log), = calls(host_library, ["gf_wkv6_prefill", ["p"] * 8 + [1, 3, H, 64, None], [0, 0]])
    assert s == 0 and len(log) == 1
    assert log[0].startswith("grid 148 " if streamed else "grid %d " % H), log


def key_compress(rows, D, Dc):
    return ["gf_gold_key_compress", ["p", "p", "p", {"ll": rows}, D, Dc, None]]


@pytest.mark.parametrize("status", [9, 701, 912])          # invalid configuration, out of resources, invalid cluster size
def test_key_compression_without_clusters(host_library, status):
    # where no cluster can be placed (a partitioned device) a short call runs on whole tiles instead of failing
    (s, log), (s1, log1) = calls(host_library, key_compress(658, 2048, 128) + [[status, 0]], key_compress(658, 2048, 128) + [[0, 0]])
    assert s1 == 0 and len(log1) == 1 and " cluster 8 " in log1[0]
    assert s == 0
    assert "refused" in log[0] and " cluster 8 " in log[0]
    assert len(log) == 2 and "refused" not in log[1] and log[1].startswith("grid 6 cluster 1 ")


def test_nothing_is_thrown_for_want_of_random_numbers(host_library):
    # a cut prefill announces its states by a number of its own; no exception may cross the C interface while it is drawn
    (s, log), (s1, log1) = calls(host_library, *[["gf_wkv6_prefill", ["p"] * 8 + [5, 700, 32, 64, None], [0, refused]] for refused in (0, 720)])
    assert s == 0 and len(log) == 1 and " cooperative " in log[0]
    # and where such a launch does not fit (cudaErrorCooperativeLaunchTooLarge) the call runs whole units
    assert s1 == 0 and len(log1) == 2 and "refused" in log1[0] and "cooperative" not in log1[1]


@pytest.mark.parametrize("status", [9, 701, 912])
def test_fp32_prefill_without_clusters(host_library, status):
    # few units: blocks of tokens over the CTAs of a cluster; where none can be placed, the same grid of columns one CTA each
    call = ["gf_wkv6_prefill_f32", ["p"] * 8 + [1, 256, 4, 64, None]]
    (s, log), (s1, log1) = calls(host_library, call + [[status, 0]], call + [[0, 0]])
    assert s1 == 0 and len(log1) == 1 and log1[0].startswith("grid 128 cluster 4 ")
    assert s == 0 and len(log) == 2 and "refused" in log[0] and log[1].startswith("grid 32 cluster 1 ")


@pytest.mark.parametrize("T,grid", [(1, 4), (4, 4), (5, 32)])
def test_fp32_prefill_of_a_few_tokens_is_not_split(host_library, T, grid):
    (s, log), = calls(host_library, ["gf_wkv6_prefill_f32", ["p"] * 8 + [1, T, 4, 64, None], [0, 0]])
    assert s == 0 and len(log) == 1 and log[0].startswith("grid %d cluster 1 " % grid), log


@pytest.mark.parametrize("chunks,c2,classic", [(8, 216, 216), (16, 240, 240), (31, 240, 240), (32, 256, 240), (63, 256, 240), (64, 256, 248), (128, 256, 248)])
def test_gradient_units_are_cut_where_that_was_measured_to_pay(host_library, chunks, c2, classic):
    # two rounds of 148 SMs, 0.27 to 0.05 of the second idle: the most units that are cut
    units = (216, 232, 240, 248, 256, 264, 280)
    logs = calls(host_library, *[backward(f, u // 8, 64 * chunks, 8, 1 << 40) + [[0, 0]] for f in (True, False) for u in units])
    cut = [any(" cooperative " in line for line in log) for s, log in logs]
    assert cut == [u <= most for most in (c2, classic) for u in units], cut

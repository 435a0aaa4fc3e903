"""The chain kernel's waits run out one at a time, on the host: its own source with every thread a coroutine and its barriers modelled
(chain_host/run.cpp).  Whichever wait of whichever warp gives up, and whichever copy never lands, every CTA has to end by itself, use its barriers
rightly and report."""
import os
import re
import subprocess
from concurrent.futures import ThreadPoolExecutor

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2504_00492_b200", "csrc")
# what a wait or an arrival is in instructions of its own, and what it is here
REDIRECTED = {"commit_at": "host::mbar_arrive(bar);", "named_arrive": "host::named(id, nthreads, false);", "add_release_gpu": "*p += v;"}
# run.cpp's configurations: d_v and a name
CONFIGS = [(128, "128x128 r=2"), (64, "64x64 r=1"), (64, "128x64 r=3"), (128, "128x128 r=1, shared out"), (64, "64x64 r=4, shared out")]


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    out = tmp_path_factory.mktemp("chain_host")
    with open(os.path.join(CSRC, "pf_chain.cu")) as f:
        source = f.read()
    source = re.sub(r"extern __shared__ __align__\(\d+\) uint8_t (\w+)\[\];", r"uint8_t* \1 = host_smem;", source)
    for name, body in REDIRECTED.items():
        source, n = re.subn(r"(void %s\([^)]*\)) \{.*?\}\n" % name, r"\1 { %s }\n" % body, source, flags=re.S)
        assert n == 1, name
    (out / "chain.inc").write_text(source)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-O1", "-w", "-fpermissive", "-I", str(out), "-I", os.path.join(HERE, "chain_host"), "-I", CSRC,
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(cuda, "include"), os.path.join(HERE, "chain_host", "run.cpp"), "-o", str(out / "run"),
                    "-Wl,--unresolved-symbols=ignore-all"], check=True)
    return str(out / "run")


@pytest.mark.parametrize("config", range(len(CONFIGS)), ids=[name for _, name in CONFIGS])
def test_every_cta_ends_whichever_wait_runs_out(program, config):
    chain = [warp for warp in range(8) if warp % 4 < CONFIGS[config][0] // 32]      # (the chain's warps that hold rows of the state)
    def ends(*args):
        r = subprocess.run([program, str(config), *map(str, args)], capture_output=True, text=True, timeout=60)
        assert r.returncode == 0, (args, r.stdout)
        return int(re.fullmatch(r"status (\d+)\n", r.stdout).group(1))

    assert ends() == 0
    with ThreadPoolExecutor(os.cpu_count()) as pool:
        # (the warps that watch mbarriers: the chain's, and those that issue products and copies; a wait past a warp's last is none)
        for warp in (*chain, *range(24, 28)):
            codes = list(pool.map(lambda n: ends(warp, n), range(64)))
            waits = sum(c != 0 for c in codes)
            assert 0 < waits < 64 and all(codes[:waits]), (warp, codes)
        assert all(pool.map(lambda n: ends("copy", n), range(3)))

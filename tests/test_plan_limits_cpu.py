"""Plans at the limit of the partial-sum buffer (no GPU): a block whose j-chunks do not fit
it gets one chunk, so that it is evaluated at all, and every plan's items cover the block."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"
TJ, THREADS = 256, 128


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.isdir(CUDA_INC):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("plan") / "plan_force_probe")
    subprocess.run(["g++", "-std=c++17", "-O1", "-x", "c++", "-I", CUDA_INC, "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_1207_2367_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "plan_force_probe.cpp"), "-o", exe], check=True)

    def run(n, m, tpi=0, jsplit=0):
        ntiles = -(-n // TJ)
        pcap = min(max(4 * n, 1 << 20), ntiles * n)          # as a context sizes it
        out = subprocess.run([exe], input=f"{ntiles} {pcap} {tpi} {jsplit} {m}\n", capture_output=True, text=True,
                             check=True).stdout
        p = dict(zip(("tpi", "ti", "tps", "b", "items"), map(int, out.split())))
        assert p["ti"] == THREADS // p["tpi"] and p["tps"] * p["b"] >= ntiles > p["tps"] * (p["b"] - 1)
        assert p["items"] == -(-m // p["ti"]) * p["b"]
        assert p["b"] == 1 or p["b"] * m <= pcap
        return p
    return run


@pytest.mark.parametrize("n,jsplit", [(262144 + 1, 5), (300000, 8), (1 << 20, 64), ((1 << 20) + 1, 5), (1 << 23, 16)])
def test_forced_split_beyond_the_buffer(plan, n, jsplit):
    fits = 4 * n // jsplit
    assert plan(n, fits, jsplit=jsplit)["b"] == -(-(-(-n // TJ)) // -(-(-(-n // TJ)) // jsplit))
    for m in (n, fits + 4 * jsplit):
        p = plan(n, m, jsplit=jsplit)
        assert (p["b"], p["tpi"]) == (1, 1)
        assert plan(n, m, tpi=4, jsplit=jsplit)["b"] == 1


@pytest.mark.parametrize("n", [1, 255, 257, 65536, (1 << 20) + 1, 8388608, 8388609, 40000000])
def test_unforced_plans_cover_every_block(plan, n):
    for m in {1, 2, max(1, n // 7), max(1, n - 1), n}:
        plan(n, m)

"""The tri-gram store's insertion code itself (csrc/tg_store.cuh), compiled for the host and run under random interleavings of its
atomic steps: the pool is never written past its end, the limit on units is exact, and nothing that nobody inserted is visible."""
import os
import re
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
STORE = os.path.join(os.path.dirname(HERE), "paper_2407_12021_b200", "csrc", "tg_store.cuh")


def _host_header(spins: int) -> str:
    """Layout and insertion, with loads that give way and a short spin limit."""
    src = open(STORE).read()
    src = src[:src.index("// ---- lookup")].replace("#pragma once", "").replace('#include "aded_internal.cuh"', "") + "}\n"
    src, n = re.subn(r'asm volatile\("ld\.acquire[^;]*;[^;]*;', "v = model_load(p);", src)
    assert n == 2
    src, n = re.subn(r'asm volatile\("st\.release[^;]*;[^;]*;', "model_store(p, v);", src)
    assert n == 1
    src, n = re.subn(r'asm volatile\("atom\.release[^;]*;[^;]*;', "seen = atomicCAS(link, 0u, base);", src)
    assert n == 1
    src, n = re.subn(r"\*reinterpret_cast<volatile (unsigned long long|uint32_t)\*>\(([^;]*?)\)(?=[;,) ])", r"model_load((\1*)(\2))", src)
    assert n == 5, n
    src, n = re.subn(r"constexpr int TG_MAX_SPIN = [^;]*;", f"constexpr int TG_MAX_SPIN = {spins};", src)
    assert n == 1
    assert "asm" not in src and "volatile" not in src
    return src


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    def build(spins):
        out = tmp_path_factory.mktemp("tg_store")
        (out / "tg_store_host.h").write_text(_host_header(spins))
        exe = out / "tg_store_host"
        subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-I", str(out), os.path.join(HERE, "tg_store_host.cpp"), "-o", str(exe)], check=True)
        return str(exe)
    return build


@pytest.mark.parametrize("chained", ["0", "1"])
def test_random_interleavings_stay_inside_the_pool_and_the_limit(program, chained):
    exe = program(1 << 20)
    for seed in range(4):
        res = subprocess.run([exe, str(seed), "100", "0", chained], capture_output=True, text=True, timeout=600)
        assert res.returncode == 0, res.stdout + res.stderr
        assert "0 timed out" in res.stdout


@pytest.mark.parametrize("chained", ["0", "1"])
def test_waits_that_run_out_leave_nothing_unwritten_in_sight(program, chained):
    """Threads held back for longer than the others wait for them: reported, and every visible entry is one that was inserted,
    counted no more often than it was."""
    exe = program(6)
    timed_out = 0
    for seed in range(4):
        res = subprocess.run([exe, str(seed), "100", "1", chained], capture_output=True, text=True, timeout=600)
        assert res.returncode == 0, res.stdout + res.stderr
        timed_out += int(res.stdout.split()[-3])
    assert timed_out > 20, "the waits did not run out"

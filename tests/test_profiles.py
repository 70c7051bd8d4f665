"""The recorded profiles: commands that end by themselves on a shared GPU, and kernels that still run.

A capture of counters replays each launch once per pass, so it names one kernel and a few launches; a launch
list (gpu__time_duration.sum alone) takes one pass and may be long.
"""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PDIR = os.path.join(ROOT, "profiles")
FILES = sorted(f for f in os.listdir(PDIR) if f.endswith(".md"))


def test_captures_of_counters_are_narrow():
    seen = 0
    for f in FILES:
        for block in re.findall(r"```\n(.*?)```", open(os.path.join(PDIR, f)).read(), flags=re.S):
            for cmd in re.findall(r"ncu .*", block.replace("\\\n", " ")):
                seen += 1
                metrics = re.findall(r"--metrics (\S+)", cmd)
                if metrics == ["gpu__time_duration.sum"] and "--set" not in cmd and "--section" not in cmd:
                    continue
                count = re.search(r" -c (\d+)", cmd)
                assert re.search(r" -k \S+", cmd) and count and int(count.group(1)) <= 3, (f, cmd)
    assert seen


def test_profiled_kernels_exist():
    csrc = os.path.join(ROOT, "paper_1205_6113_gb300", "csrc")
    source = "".join(open(os.path.join(csrc, f)).read() for f in sorted(os.listdir(csrc)) if f.endswith((".cu", ".cuh")))
    kernels = set(re.findall(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(", source))
    for f in FILES:
        for name in re.findall(r"`(k[bk]?_\w+)[<`]", open(os.path.join(PDIR, f)).read()):
            if name.endswith("_"):
                continue                                          # a family, kk_*
            assert name in kernels, (f, name)

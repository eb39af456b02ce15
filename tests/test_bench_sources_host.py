"""The sources whose hash ties bench.py's committed counters to the headline
kernel: every header that the kernel is built from, and the counters name an
instance that those sources launch."""
import importlib.util
import json
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = "paper_2508_16121_gb300/csrc"


def _bench():
    spec = importlib.util.spec_from_file_location("bench_src", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def _headers(name, seen):
    with open(os.path.join(ROOT, CSRC, name)) as f:
        for h in re.findall(r'#include "(apply_\w+\.cuh)"', f.read()):
            if h not in seen:
                seen.add(h)
                _headers(h, seen)
    return seen


def test_the_hash_covers_the_headline_kernel():
    b = _bench()
    for h in _headers("apply_f32_16.cu", set()):
        assert f"{CSRC}/{h}" in b.KERNEL_SOURCES, h


def test_the_counters_name_an_instance_of_the_kernel():
    b = _bench()
    with open(os.path.join(ROOT, b.PROFILE_COUNTERS)) as f:
        name = json.load(f)["kernel"]
    with open(os.path.join(ROOT, CSRC, "apply_kernel.cuh")) as f:
        decl = re.search(r"template <([^<>]*)>\s*__global__ void __launch_bounds__\(kThreads, 1\) apply_kernel", f.read())
    args = re.match(r"apply_kernel<Io<InF32, OutF32>, (.*)>$", name)
    assert args and len(args.group(1).split(",")) == len(decl.group(1).split(",")) - 1, name
    assert name in open(os.path.join(ROOT, "bench.py")).read()

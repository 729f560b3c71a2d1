"""What the bench says about the library's kernels agrees with the library's sources."""
import os
import re
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402

CSRC = os.path.join(ROOT, "paper_2405_12913_gb300", "csrc")


def _read(name):
    return open(os.path.join(CSRC, name), encoding="utf-8").read()


@pytest.mark.parametrize("phase", ["ray_step", "kspace"])
def test_a_record_depends_on_every_file_with_device_code(phase):
    # the .cu files of a phase, and of the headers that they include, at any depth, those with device functions; a file
    # that instantiates templates of one of those headers too
    listed = bench.KERNEL_SOURCES[phase]
    todo, seen = [f for f in listed if f.endswith((".cu", ".cuh"))], set()
    while todo:
        f = todo.pop()
        if f in seen:
            continue
        seen.add(f)
        todo += [h for h in re.findall(r'#include "([a-z_]+\.c?u?h)"', _read(f)) if os.path.exists(os.path.join(CSRC, h))]
    device = {f for f in seen if "__device__" in _read(f) or "__global__" in _read(f)}
    templates = [f for f in listed if f.endswith(".cuh") and "template <int R1>" in _read(f)]
    for f in os.listdir(CSRC):
        if f.endswith(".cu") and any(f'#include "{t}"' in _read(f) for t in templates):
            device.add(f)
    assert device <= set(listed), device - set(listed)


def test_the_bench_knows_the_sides_of_the_FFT_passes():
    body = _read("fft_passes.cu").split("bool fft_supported(int64_t n) {")[1].split("}")[0]
    sides = {int(x) for x in re.findall(r"case (\d+):", body)}

    class W:
        n_mesh = 0

    assert len(sides) >= 9
    for n in range(2, 2049, 2):
        W.n_mesh = n
        assert bench.own_fft(W) == (n in sides), n

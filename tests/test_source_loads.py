"""What the kernels may read through the read-only path.  Kernels launched with launch_after are resident before the kernel ahead of them has
ended; what that one writes (positions, velocities, forces, totals, flags) changes during their lifetime, which the read-only path
does not allow.  Results cannot show a stale line reliably, so the sources are looked at."""
import glob
import os
import re

import pytest

from conftest import ROOT

SOURCES = {os.path.basename(p): open(p).read() for p in sorted(glob.glob(os.path.join(ROOT, "paper_2608_16329_b200", "csrc", "*.cu*")))}
EXCHANGED = r"pos4|pos\b|vel\b|force|disp|acc|status|far_flag|rebuild_flag|tile_counter|pair_counter|block_sum|scale\b|e_atom|stamp"


def _kernels_launched_early():
    names = set()
    for text in SOURCES.values():
        for args in re.findall(r"launch_after(?:_if)?\((.*?)\)\);", text, flags=re.S):
            names.update(re.findall(r"\bk_\w+", args))
    return names


@pytest.mark.parametrize("name", sorted(SOURCES))
def test_moving_data_is_not_loaded_as_read_only(name):
    text = re.sub(r"//[^\n]*", "", SOURCES[name])
    early = _kernels_launched_early()
    assert {"k_kick_drift", "k_set_positions", "k_outputs", "k_kinetic"} <= early
    for expr in re.findall(r"__ldg\(([^;]*)\)", text):
        assert not re.match(r"\s*&?(k\.|k->)?(%s)" % EXCHANGED, expr), expr
    for kernel, params in re.findall(r"__global__[^;{]*?\b(k_\w+)\((.*?)\)\s*\{", text, flags=re.S):
        if kernel in early:
            for param in re.findall(r"const [\w:]+ \*__restrict__ (\w+)", params):
                assert not re.fullmatch(EXCHANGED, param), (kernel, param)
    for function, body in re.findall(r"__device__ __forceinline__ \w+ (load_\w+)\(.*?\)\s*\{(.*?)\n\}", text, flags=re.S):
        assert ".nc." not in body, function

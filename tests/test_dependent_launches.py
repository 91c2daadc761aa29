"""Kernels launched before their predecessor on the stream has ended (programmatic dependent launch) and waiting for it on
the device must not promise, by ``__restrict__`` or a read-only load, that nothing writes their inputs while they live: the
predecessor still does. Read from the sources."""
import glob
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1009_2727_gb300", "csrc")
WAIT = re.compile(r"\b(chain_wait|cudaGridDependencySynchronize)\s*\(\s*\)")


def block(s, i, o, c):
    """the text from the first `o` at or after i to the `c` that closes it"""
    i = s.index(o, i)
    d = 0
    for j in range(i, len(s)):
        d += (s[j] == o) - (s[j] == c)
        if d == 0:
            return s[i:j + 1], j + 1
    raise AssertionError("unbalanced")


def kernels():
    out = []
    for f in sorted(glob.glob(os.path.join(SRC, "*.cu"))):
        s = re.sub(r"//[^\n]*", "", open(f).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__)?", s):
            i = m.end()
            if m.group(0).rstrip().endswith("__launch_bounds__"):
                _, i = block(s, i, "(", ")")
            name = re.match(r"\s*(\w+)", s[i:]).group(1)
            par, i = block(s, i, "(", ")")
            body, _ = block(s, i, "{", "}")
            out.append((os.path.basename(f), name, par, body))
    return out


WAITING = [k for k in kernels() if WAIT.search(k[3])]


def test_the_waiting_kernels_are_found():
    names = {k[1] for k in WAITING}
    assert {"k1_push", "k3_ampere", "k3_faraday_few", "k3_filter_zs", "k_push", "k_sb_fwd"} <= names and len(names) > 25


@pytest.mark.parametrize("k", WAITING, ids=lambda k: f"{k[0]}-{k[1]}")
def test_waiting_kernel_takes_plain_pointers(k):
    _, name, par, body = k
    assert "__restrict__" not in par, name
    assert "__ldg(" not in body and "ld.global.nc" not in body, name


def test_the_push_starts_on_idle_sms():
    """its shared memory and L1 are split when a kernel finds an SM idle: started beside the filter's blocks, the push and
    its global-memory pass have a sixth of their L1 (a heated stage takes 2.5 ms a step instead of 1.8)"""
    src = re.sub(r"//[^\n]*", "", open(os.path.join(SRC, "pic_particles.cu")).read())
    assert not re.search(r"launch_chained\(\s*k_push(_batch)?\s*<", src)
    assert re.search(r"k_push<T, 3, false>\s*<<<", src) and re.search(r"k_push_batch<T, 3>\s*<<<", src)

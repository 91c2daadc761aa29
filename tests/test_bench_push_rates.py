"""The bench's push rates count the particles that a step pushed: resting chunks are neither read nor written, and the DRAM
traffic is a figure of steps in which every particle is pushed and does not fit in L2."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_resting_particles_are_not_charged():
    # 13.2 million electrons of which 1.2 million are pushed in 0.1 ms: 60 bytes each
    r = bench.push_roofline(1.2e6, 12e6, 0.1, 60, 49.6, 6784.0)
    assert r["achieved"] == pytest.approx(1.2e6 * 60 / 1e-4 / 1e9) and r["frac"] < 0.2
    assert r["traffic"] is None
    assert (r["particles_pushed_per_step"], r["particles_at_rest_per_step"]) == (1.2e6, 12e6)


def test_traffic_only_where_it_was_measured():
    assert bench.push_roofline(13.2e6, 0.0, 0.37, 60, 49.6, 6784.0)["traffic"] == pytest.approx(49.6 * 13.2e6)
    assert bench.push_roofline(13.2e6, 0.0, 0.37, 60, None, 6784.0)["traffic"] is None
    assert bench.push_roofline(1e6, 0.0, 0.03, 60, 49.6, 6784.0)["traffic"] is None       # fits in L2


def test_instruction_constants_are_of_pushed_particles():
    # a particle's gather, push and deposit are hundreds of operations; an average over resting ones was 42.7
    assert bench.PUSH_WARP_INST_PER_PARTICLE > 15 and bench.PUSH_FLOPS_PER_PARTICLE > 150


def test_every_name_is_defined():
    """the bench's modes mostly run on a GPU only: no function may read a global that the module has not"""
    import builtins
    import dis
    import types

    def functions(code):
        yield code
        for c in code.co_consts:
            if isinstance(c, types.CodeType):
                yield from functions(c)

    code = compile(open(bench.__file__).read(), "bench.py", "exec")
    missing = {(f.co_name, i.argval) for f in functions(code) for i in dis.get_instructions(f)
               if i.opname in ("LOAD_GLOBAL", "LOAD_NAME") and f is not code
               and not hasattr(bench, i.argval) and not hasattr(builtins, i.argval)}
    assert not {m for m in missing if not m[1].startswith("__")}, missing

"""Rules the CUDA sources keep, read from the sources themselves (what they guard against shows on a GPU only now and
then, or not with today's compiler)."""
import os
import random
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0808_3510_gb300", "csrc")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        s = f.read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", s, flags=re.S))


def _kernels(code):
    """(name, parameter list) of every __global__ function."""
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\(\d+\)\s*)?(\w+)\(([^)]*)\)", code):
        yield m.group(1), m.group(2)


@pytest.mark.parametrize("name", SOURCES)
def test_read_only_loads_are_of_plan_tables(name):
    """A kernel launched as a programmatic dependent begins before the previous one ends: what that one may have
    written must not be loaded as data that is constant while the kernel runs."""
    code = _code(name)
    tables = r"(tw|prescale|P\.zt|tab|P\.model_tab)\["
    for m in re.finditer(r"__ldg\(([^;]*)", code):
        arg = m.group(1)
        assert re.match(r"&" + tables, arg) or re.match(r"T \+ ", arg), f"{name}: __ldg({arg[:40]}"
    for kernel, params in _kernels(code):
        for p in params.split(","):
            if "__restrict__" in p and "const" in p:
                assert p.split()[-1] == "tw", f"{name}: {kernel}: {p.strip()}"


@pytest.mark.parametrize("name", SOURCES)
def test_dynamic_shared_memory_is_aligned_for_16_byte_cells(name):
    """Row slots hold 16-byte cells and node records at offsets that are multiples of 16: the base has to be one."""
    for m in re.finditer(r"extern\s+__shared__([^;]*);", _code(name)):
        assert "__align__(16)" in m.group(1), f"{name}: extern __shared__{m.group(1)}"


@pytest.mark.parametrize("nitems,ctas,launches", [(2, 1, 1), (40, 7, 1), (2, 1, 2), (5, 4, 2), (40, 7, 2), (40, 7, 3), (301, 152, 2)])
def test_work_counter_is_zero_after_overlapping_launches(nitems, ctas, launches):
    """The row kernels draw work items from a counter that no launch sets beforehand: it has to be zero after every
    launch, and after launches that overlapped in any order, or the next call would leave out rows."""
    code = _code("pai_row_kernels.cuh")
    uses = re.findall(r"\bL\.counter\b[^;]*", code)
    assert len(uses) == 1 and uses[0].startswith("L.counter, (unsigned)(L.nitems - 1))")
    assert "gridDim.x + atomicInc(L.counter" in code
    for seed in range(20):
        rng = random.Random(seed)
        counter, done = 0, [set(range(ctas)) for _ in range(launches)]  # the first items are the block indices
        running = [(k, c) for k in range(launches) for c in range(ctas)]
        while running:
            i = rng.randrange(len(running))
            ticket, counter = counter, 0 if counter >= nitems - 1 else counter + 1  # atomicInc
            if ctas + ticket < nitems:
                done[running[i][0]].add(ctas + ticket)
            else:
                running.pop(i)
        assert counter == 0
        assert launches > 1 or done[0] == set(range(nitems))


def test_every_device_function_is_used():
    code = "".join(_code(f) for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh", ".h", ".cpp")))
    for name in set(re.findall(r"__device__\s+__forceinline__\s+[\w:<>, ]*?[&*]?\s(\w+)\(", code)):
        assert len(re.findall(rf"\b{name}\b", code)) > 1, name

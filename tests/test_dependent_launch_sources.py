"""Rules of the kernels that may start before the kernel before them has
finished (pdl.cuh), checked in the sources: a race there would show only now
and then.  Runs without a GPU."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1610_04914_gb300", "csrc")


def kernels():
    """(name, parameters, body) of every __global__ function that waits, in its
    own body, for the kernel before it."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
        for m in re.finditer(r"__global__[^;{]*?(k_\w+)\s*\(([^{]*)\)\s*\{", text):
            depth, at = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[at], 0)
                at += 1
            if "pdl_wait()" in text[m.end():at]:
                out.append((m.group(1), m.group(2), text[m.end():at]))
    return out


def test_kernels_are_found():
    names = {k[0] for k in kernels()}
    assert {"k_pulse_f32", "k_pulse_batch", "k_obs_partial", "k_obs_final", "k_stage32", "k_stage64", "k_metropolis",
            "k_step_rk5", "k_adj_xw"} <= names


def test_pulse_number_is_read_after_the_wait():
    """The pulse number is written by an earlier kernel: a plain load of it
    stands after the wait, and a kernel that draws before (with
    load_shared_word, a value that may be old) reads it again afterwards."""
    for name, _, body in kernels():
        before, after = body.split("pdl_wait()", 1)
        assert not re.search(r"\*\s*(a\.)?interval\b", before), name
        if "load_shared_word" in before:
            assert "load_shared_word" in after, name


def test_data_of_earlier_kernels_is_read_by_plain_loads():
    """A load that the compiler takes for one of unchanging data may move ahead
    of the wait: only the constant tables are read that way."""
    for name, params, _ in kernels():
        assert not re.search(r"const\s+(real|float|double|long long)\s*\*\s*__restrict__", params), name
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        assert all(t.startswith("&k") for t in re.findall(r"__ldg\(([^)]*)", text)), path
    for header in ("patch_tile.cuh", "step_rk5.cu"):
        text = open(os.path.join(CSRC, header)).read()
        assert not re.search(r"const float\*\s*__restrict__", text), header

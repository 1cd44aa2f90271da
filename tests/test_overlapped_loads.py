"""Reads of kernels that overlap the one before them on the stream (CPU check of
the sources): each begins with the wait, hands it every pointer that it could
read through the read-only path, and uses explicit read-only loads only on data
that the kernel before it does not write."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2103_05162_gb300", "csrc")


def kernels():
    """(name, parameters, body) of every kernel."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        with open(path) as f:
            s = f.read()
        for m in re.finditer(r"__global__\s+void\s+(?:__\w+\([^{]*?\)\s*)?(\w+)\s*\(", s):
            end, depth = m.end(), 1
            while depth:
                depth += {"(": 1, ")": -1}.get(s[end], 0)
                end += 1
            body = s[s.index("{", end):]
            yield m.group(1), s[m.end():end - 1], body[1:body.index("\n}\n")]


def test_kernels_begin_with_the_wait_and_hand_it_their_inputs():
    seen = 0
    for name, params, body in kernels():
        if name == "k_count_phase":  # (counters build, launched plainly)
            continue
        first = re.match(r"\s*stage_begin\(([^)]*)\);", body)
        assert first, f"{name} does something before the wait"
        given = {a.strip() for a in first.group(1).split(",")}
        inputs = set(re.findall(r"const\s+[\w:<> ]*?\*\s*__restrict__\s+(\w+)", params))
        assert inputs <= given, f"{name}: {sorted(inputs - given)} may be read through the read-only path"
        seen += 1
    assert seen > 30


def test_read_only_loads_are_of_older_data():
    # the caller's points and offsets, nodes and leaf records (refit and leaf
    # kernels, with the initialisation and the lists in between)
    older = r"__ldg\((reinterpret_cast<const float[24]\*>\()?(pts|offs|&n\[i\]|&a\.leafr\[)"
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        with open(path) as f:
            code = re.sub(r"//.*", "", f.read())
        for m in re.finditer(r"__ldg\([^;]*", code):
            assert re.match(older, m.group(0)), f"{os.path.basename(path)}: {m.group(0)}"


def test_device_functions_take_plain_pointers_to_newer_data():
    # const __restrict__ is left to the caller's points and offsets and to the
    # traversals' boxes
    found = set()
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        with open(path) as f:
            s = f.read()
        for m in re.finditer(r"__device__ [^;{}()]*?(\w+)\(([^{};]*?)\)\s*(?:const)?\s*\{", s):
            names = set(re.findall(r"const\s+[\w:<> ]*?\*\s*__restrict__\s+(\w+)", m.group(2)))
            assert names <= {"pts", "p", "offs", "boxes"}, f"{os.path.basename(path)}: {m.group(1)}: {sorted(names)}"
            found |= names
    assert found == {"pts", "p", "offs", "boxes"}

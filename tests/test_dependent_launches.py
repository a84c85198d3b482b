"""Kernels launched behind one another (pdl_wait) may start while the kernel before
them still writes, so what an earlier kernel of the library wrote is read by plain
loads: __ldg and `const ... __restrict__` promise data that nothing writes while the
kernel lives.  Checked in the sources, over every function that such a kernel calls;
only the inputs that no kernel of the library writes may be read that way."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1911_12070_gb300", "csrc")
INPUTS = {"psi", "X", "T"}  # the field, training rows and targets


def _functions(src):
    """name -> (parameters, body) of the functions at namespace level."""
    src = re.sub(r"//[^\n]*", "", src)
    out, depth, start = {}, 0, 0
    for m in re.finditer(r"[{}]", src):
        head = src[start:m.start()]
        if m.group() == "{":
            if re.search(r"namespace(\s+\w+)?\s*$", head) or re.search(r'extern "C"\s*$', head):
                start = m.end()
                continue
            if depth == 0:
                opened, begin = head.split(";")[-1], m.end()
            depth += 1
        elif depth > 0:
            depth -= 1
            if depth == 0:
                called = [n for n in re.findall(r"(\w+)\s*\(", opened) if not n.startswith("__")]
                if called:
                    out[called[0]] = (opened, src[begin:m.start()])
                start = m.end()
        else:
            start = m.end()
    return out


FILES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


@pytest.fixture(scope="module")
def functions():
    return {f: _functions(open(os.path.join(CSRC, f)).read()) for f in FILES}


def _reached(functions, file, name):
    """(file, name) of a kernel and of what it calls in its file and the headers."""
    todo, seen = [name], {}
    while todo:
        n = todo.pop()
        for f in [file] + [h for h in FILES if h.endswith("h")]:
            if n in functions[f] and (f, n) not in seen:
                seen[f, n] = functions[f][n]
                todo += re.findall(r"\b(\w+)\s*(?:<[^<>;]*>)?\(", functions[f][n][1])
    return seen


def test_written_data_is_read_by_plain_loads(functions):
    kernels = [(f, n) for f in FILES for n, (_, b) in functions[f].items() if "pdl_wait();" in b]
    assert {"expand_bits_kernel", "localize_kernel", "train_rows_kernel", "train_grads_kernel",
            "train_update_kernel", "adjacency_kernel", "reduce_init_kernel", "orient_kernel",
            "v3_scan_kernel"} <= {n for _, n in kernels}
    wrong = set()
    for file, kernel in kernels:
        for (f, n), (params, body) in _reached(functions, file, kernel).items():
            const = re.findall(r"const\s[^,;()]*__restrict__\s+(\w+)", params + body)
            wrong |= {(f, n, p) for p in const if p not in INPUTS}
            for arg in re.findall(r"__ldg\(\s*([^;]*)", body):
                base = re.match(r"[&(]*\s*(?:reinterpret_cast<[^>]*>\()*\s*(?:\w+\.)?(\w+)", arg)
                if base.group(1) not in INPUTS:
                    wrong.add((f, n, arg[:40]))
    assert not wrong, sorted(wrong)

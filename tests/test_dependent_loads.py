"""Kernels that may be launched as programmatic dependents start while the
kernel before them still runs, so nothing that a kernel of the call wrote may be
read by non-coherent loads (__ldg), which are for memory nobody writes during a
kernel's life and which no wait orders. Read from the sources: such a load takes
K or V rows only (the call's inputs)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2607_22586_gb300", "csrc")
INPUT_LOADS = {
    "score_simt.cu": ["if constexpr (INPUT) return __ldg(p)"],
}


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _overlapped():
    return [n for n in sorted(os.listdir(CSRC)) if n.endswith(".cu") and "dependent_start();" in _code(n)]


def test_only_inputs_by_non_coherent_loads():
    files = _overlapped()
    assert {"proxy.cu", "score_simt.cu", "score_umma.cu", "select.cu"} <= set(files)
    for name in files:
        code = _code(name)
        for load in INPUT_LOADS.get(name, []):
            assert code.count(load) == 1, (name, load)
            code = code.replace(load, "")
        for load in re.findall(r"load_row16\(([^)]*)\)", code):
            assert name == "select.cu" and re.match(r"[KV] \+ src", load), (name, load)
        assert "__ldg" not in code and "ld.global.nc" not in code and "__restrict__" not in code, name


def test_cuda_core_tiles_of_inputs_are_those_of_K():
    # Piece<element, rows, dimensions, INPUT>: key tiles from K, proxy tiles from
    # the packed block
    pieces = re.findall(r"Piece<T, (T[KR]), KC, (true|false)> \w+;", _code("score_simt.cu"))
    assert sorted(pieces) == [("TK", "true"), ("TK", "true"), ("TR", "false"), ("TR", "false")]

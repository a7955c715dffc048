"""The form in which the kernels issue tensor-core instructions, by reading the
sources: tcgen05.mma and tcgen05.commit are for one elected thread of a
converged warp, so every branch that holds them is warp-uniform and elects its
thread, and the kind of an MMA (FP16 or E4M3) is a template parameter, so that
no branch holds two kinds chosen at run time."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_17770_gb300", "csrc")


def _issuing_lines():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        lines = [re.sub(r"//.*", "", l) for l in open(path).read().split("\n")]
        for i, line in enumerate(lines):
            if re.search(r"\btc::(mma_\w+|commit)\(", line):
                yield os.path.basename(path), i, line, lines


def _branch(lines, i):
    """The innermost `if (...) {` around line i, loops left out."""
    depth = 0
    for k in range(i - 1, -1, -1):
        depth += lines[k].count("}") - lines[k].count("{")
        if depth < 0:
            if re.match(r"\s*for \(", lines[k]):
                depth = 0
                continue
            return lines[k].strip()
    return ""


def test_one_elected_thread_issues_every_mma():
    found = list(_issuing_lines())
    assert len(found) >= 30
    for name, i, line, lines in found:
        assert _branch(lines, i) == "if (warp == 0 && tc::elect_one()) {", (name, i + 1, _branch(lines, i))


def test_the_kind_of_an_mma_is_a_template_parameter():
    for name, i, line, lines in _issuing_lines():
        m = re.match(r"\s*if \((\w+)\) tc::mma_", line)
        assert m is None or m.group(1) == "kFp8", (name, i + 1, line)
        if re.match(r"\s*else tc::mma_", line):
            assert re.match(r"\s*if \(kFp8\) tc::mma_", lines[i - 1]), (name, i + 1, lines[i - 1])


def test_the_issuing_warp_is_known_to_be_uniform():
    for name in {f[0] for f in _issuing_lines()}:
        src = open(os.path.join(CSRC, name)).read()
        decl = re.findall(r"const int warp = ([^;]+);", src)
        assert any("__shfl_sync(FULL" in d for d in decl), name

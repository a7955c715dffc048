"""The debug build's index checks, by reading the sources: in the kernels of
the learned decode every access to a row's value, and every access to the
texel list and the outputs of ctf_mlp_decode, goes through ck (directly, or
through row_of, which does)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_17770_gb300", "csrc")


@pytest.mark.parametrize("name,arrays", [
    ("ctf_mlp_dense.cu", ("outrow", "a.xy", "a.out")), ("ctf_mlp_ws2.cu", ("outrow",)), ("ctf_mlp_ws.cu", ("outrow",)),
    ("ctf_mlp_chain.cuh", ("outrow",))])
def test_every_access_is_checked(name, arrays):
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    for a in arrays:
        uses = re.findall(r"(?<![\w.])" + re.escape(a) + r"\[([^\n]*)", src)
        assert uses, (name, a)
        for u in uses:
            assert u.startswith("ck(") or re.match(r"row_of\((?:[^()]|\([^()]*\)|\((?:[^()]|\([^()]*\))*\))*\)\]", u), (name, a, u)

"""The push and the adjoint's recomputation of its move take 1 / gamma from one
function (no GPU needed): with a root of its own on either side, an ulp in the
new offset can put a particle on the other side of a cell face."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1503_02464_gb300", "csrc")


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def test_one_inverse_gamma():
    shared = _source("pic_device.cuh")
    assert len(re.findall(r"\bR inv_gamma\(const R u\[3\]\)", shared)) == 1
    for name in ("push.cu", "adjoint.cu"):
        text = _source(name)
        assert re.search(r"\big = inv_gamma<R>\(", text), name
        assert not re.search(r"\bfloat>?\(float x\) \{ return rsqrtf|\brsqrt\(x\)|1\.0 / sqrt\(x\)", text), name

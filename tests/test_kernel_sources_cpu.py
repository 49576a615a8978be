"""Rules of the CUDA sources that only reading can show: nothing here needs a
GPU, and a source that breaks one may well run correctly for a long time."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2606_00817_gb300", "csrc")


def _sources(pattern="*"):
    """{file name: text without comments} of csrc."""
    out = {}
    for path in sorted(glob.glob(os.path.join(CSRC, pattern))):
        text = open(path).read()
        out[os.path.basename(path)] = re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)
    assert out
    return out


def test_tensor_maps_reach_kernels_by_value():
    """A tensor map in global memory has to be acquired by the tensor-map proxy
    before it is used; a __grid_constant__ parameter has not. No structure that
    a kernel takes points at maps, no kernel has a pointer to them, and none are
    copied to the device."""
    for name, text in _sources().items():
        if "fence.proxy.tensormap" in text:
            continue
        for body in re.findall(r"\bstruct \w+ \{(.*?)\n\};", text, flags=re.S):
            assert not re.search(r"CUtensorMap\s*\*", body), name
        for args in re.findall(r"__global__.*?\((.*?)\)\s*\{", text, flags=re.S):
            assert not re.search(r"CUtensorMap\s*\*", args), name
        assert not re.search(r"cudaMemcpy\w*\([^;]*CUtensorMap", text), name

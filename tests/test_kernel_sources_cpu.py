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


def test_pair_allocations_follow_a_cluster_barrier():
    """An allocation of tensor memory for a CTA pair works on the peer too and
    waits without a limit, so every kernel first passes a cluster barrier, which
    shows that the peer has started."""
    found = 0
    for name, text in _sources("*.cu").items():
        for kernel in re.split(r"__global__", text)[1:]:
            at = kernel.find("tmem_alloc_pair(")
            if at < 0:
                continue
            found += 1
            before = kernel[:at]
            assert "cluster_sync_all()" in before or (
                0 <= before.find("cluster_arrive_relaxed()") < before.find("cluster_wait()")), name
    assert found >= 2


def test_no_cta_leaves_with_copies_in_flight():
    """A producer that has issued its last copy may leave while another role
    gives up waiting for it, so the wait for the copies in flight depends on no
    outcome: each single-CTA kernel that loads tiles ends its producer with one,
    outside of any `if (!ok) { ... }`."""
    found = 0
    for name, text in _sources("*.cu").items():
        for kernel in re.split(r"__global__", text)[1:]:
            if "tma_load_2d(" not in kernel:
                continue
            found += 1
            assert re.search(r"mbar_wait_bounded\(full_bar\([^;]*nullptr, k\w+Ns\)", kernel), name
            for block in re.findall(r"if \(!ok\) \{([^{}]*)\}", kernel):
                assert "full_bar(" not in block, name
    assert found >= 6


def test_shared_memory_limits_are_constants():
    """A kernel's limit of dynamic shared memory belongs to the function, not to a
    field or a host thread: a launcher that set it to its own field's size could
    lower it between another thread's setting and launch. Every limit is made of
    constants only."""
    found = 0
    constant = re.compile(r"k[A-Z]\w*|[A-Z][A-Z0-9_]*|[A-Z]\w*Shape|HgSmem|\w*bytes|\d+")
    for name, text in _sources("*.cu").items():
        for limit in re.findall(r"cudaFuncAttributeMaxDynamicSharedMemorySize,\s*(.*?)\)\s*(?:;|!=|==)",
                                text, flags=re.S):
            found += 1
            for word in re.findall(r"\w+", limit):
                assert constant.fullmatch(word), (name, limit)
    assert found >= 15

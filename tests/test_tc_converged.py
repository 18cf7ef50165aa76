"""The tensor-memory instructions that need a whole, converged warp
(.sync.aligned): a lane that took another branch must have been brought back
before each of them.  Checked on the source, since a warp that is not converged
there is undefined behaviour on the GPU."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1901_08269_gb300", "csrc")


def sources():
    for f in sorted(os.listdir(SRC)):
        if f.endswith((".cu", ".cuh")):
            with open(os.path.join(SRC, f)) as h:
                yield f, re.sub(r"//[^\n]*", "", h.read())


def test_aligned_instructions_are_issued_by_the_wrappers_alone():
    assert [f for f, s in sources() if ".sync.aligned" in s] == ["cfp_tc.cuh"]


def test_wrappers_reconverge_the_warp_first():
    text = dict(sources())["cfp_tc.cuh"]
    aligned = {}
    for part in text.split("__device__ __forceinline__")[1:]:
        if ".sync.aligned" in part:
            aligned[re.match(r"\s*\w+ (\w+)\(", part).group(1)] = part[part.index("{"):]
    assert set(aligned) == {"tmem_alloc", "tmem_free", "tmem_ld16"}
    for name, body in aligned.items():
        assert "__syncwarp();" in body[:body.index(".sync.aligned")], name

"""A kernel started as a dependent launch waits before it reads what its
predecessor writes.  Loads that the compiler takes for invariant (through
const __restrict__ pointers, or __ldg) are not held back by the wait's memory
clobber, only by a wait that re-defines their pointers: pdl_wait(p, ...)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2008_09441_gb300", "csrc")
# tables written once, at set-up, are no predecessor's output
INVARIANT = re.compile(r"__ldg\(|\bld4\(|const (?!\w*Job\b)\w+(<\w+>)?\* __restrict__")


def test_waits_cover_invariant_loads():
    bare = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        for body in re.split(r"^}", code, flags=re.M):
            if "pdl_wait();" in body and INVARIANT.search(body):
                bare.append(re.findall(r"\bk_\w+", body)[-1])
    assert bare == []

"""CPU reading of the kernels' TMA producers: after its last copy a producer waits (bounded) until the
MMAs have released every ring slot, so that a CTA whose MMA issuer gave up does not leave with
copies in flight, and a wait that runs out is followed by waits for the copies themselves."""
import os
import re

from paper_2606_07878_gb300 import still

CSRC = os.path.join(os.path.dirname(still.LIB_PATH), "csrc")


def _producers():
    for name in sorted(os.listdir(CSRC)):
        src = open(os.path.join(CSRC, name)).read()
        for part in re.split(r"-{20,} TMA producer", src)[1:]:
            yield name, re.split(r"-{20,} MMA issuer", part)[0]


def test_every_producer_waits_for_its_slots_and_copies():
    seen = []
    for name, body in _producers():
        seen.append(name)
        body = re.sub(r"//[^\n]*", "", body)
        closing = re.search(r"for \(int i = 0; i < kStages[^{]*\{\s*if \(!mbar_wait\(&a?empty\[stage\], "
                            r"phase \^ 1\)\) \{(.*)", body, re.S)
        assert closing, f"{name}: no wait for the ring slots behind the last copy"
        tail = closing.group(1)
        assert "tma_load" not in tail, name
        assert re.search(r"abort_flag = 1|fail\(", tail), f"{name}: a wait that runs out sets no flag"
        assert re.search(r"if \((bad \|\| )?\*abort_flag[^)]*\).*mbar_wait(_cluster)?\(&a?full\[", tail, re.S), (
            f"{name}: copies in flight are not waited for")
    assert seen.count("tc_gemm.cuh") == 3 and {"ca_flash.cuh", "ca_pair.cu", "keyproj.cuh"} <= set(seen)

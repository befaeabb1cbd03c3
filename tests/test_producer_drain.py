"""CPU reading of the kernels' TMA producers: no CTA leaves with copies in flight behind an MMA issuer
that gave up. Either the producer waits (bounded) behind its last copy until the MMAs have released
every ring slot, and then for the copies themselves, or the issuer that gives up waits for them."""
import os
import re

from paper_2606_07878_gb300 import still

CSRC = os.path.join(os.path.dirname(still.LIB_PATH), "csrc")
COPIES = r"mbar_wait(_cluster)?\(&a?full\["


def _roles():
    """(file, producer, MMA issuer) of every kernel with a TMA producer."""
    for name in sorted(os.listdir(CSRC)):
        src = re.sub(r"// [^\n-][^\n]*", "", open(os.path.join(CSRC, name)).read())
        for part in re.split(r"-{20,} TMA producer", src)[1:]:
            producer, issuer = re.split(r"-{20,} MMA issuer", part)[:2]
            yield name, producer, re.split(r"// -{20,}", issuer)[0]


def _producer_waits(producer):
    closing = re.search(r"for \(int i = 0; i < kStages[^{]*\{\s*if \(!mbar_wait\(&a?empty\[stage\], "
                        r"phase \^ 1\)\) \{(.*)", producer, re.S)
    if not closing or "tma_load" in closing.group(1):
        return False
    return bool(re.search(r"(abort_flag = 1|fail\().*if \((bad \|\| )?\*abort_flag[^)]*\).*" + COPIES,
                          closing.group(1), re.S))


def _issuer_waits(issuer):
    """A round of the ring behind the place where the issuer gives up."""
    return bool(re.search(r"abort_flag(\) \{| = 1;).*for \(int \w+ = [^;]*; \w+ < [^;]*kStages[^;]*; "
                          r"\+\+\w+\) \{\s*\(void\)" + COPIES, issuer, re.S))


def test_no_kernel_leaves_with_copies_in_flight():
    seen = []
    for name, producer, issuer in _roles():
        seen.append(name)
        assert _producer_waits(producer) or _issuer_waits(issuer), (name, len(seen))
    assert seen.count("tc_gemm.cuh") == 3 and {"ca_flash.cuh", "ca_pair.cu", "keyproj.cuh"} <= set(seen)

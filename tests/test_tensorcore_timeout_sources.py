"""What the tensor-core tiles wait for before they free their TMEM and leave.  After a timeout
every ordinary wait returns at once (it looks at the abort flag), while MMAs and copies may still
be on their way; whether they are shows in no result, so the source is checked."""
import os
import re

import pytest

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1905_00444_gb300", "csrc",
                      "cgemm_tc.cu")


def ending(kernel):
    """The code of a kernel after its roles: from its last role's end to its own."""
    text = re.sub(r"//[^\n]*", "", open(SOURCE).read())
    start = re.search(kernel + r"\(const TcArgs", text).end()
    body = text[start:text.index("\n}\n", start)]
    return body[body.rindex("\n  }\n\n") + 4:]      # roles close at this depth, before a blank line


@pytest.mark.parametrize("kernel", ["cgemm_cta_kernel", "cgemm_pair_kernel"])
def test_mmas_end_before_tmem_is_freed(kernel):
    end = ending(kernel)
    dealloc = end.index("tcgen05.dealloc")
    assert "mbar_wait(" not in end, "a wait that a timeout cuts short"
    assert re.search(r"mbar_drain\(done, 0, kWaitNs", end[:dealloc])


def test_pair_waits_for_what_the_other_cta_sends():
    """The leader's MMAs end before the cluster barrier, the other CTA sees their last commit
    before the second one, and site copies in flight after a timeout land before it."""
    end = ending("cgemm_pair_kernel")
    first, second = [m.start() for m in re.finditer(r"cluster_barrier\(\);", end)]
    assert re.search(r"rank == 0\) mbar_drain\(done", end[:first])
    assert re.search(r"mbar_drain\(done", end[first:second])
    assert re.search(r"\*abort\) \{.*mbar_drain\(rank == 0 \? full\(", end[first:second], re.S)

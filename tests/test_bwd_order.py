"""CPU-only: no product of the backward kernel overwrites tensor memory that an earlier product may still read, read
from the order of issue in their source.

Products run in their order of issue only if they share accumulator and shape.  At head_dim 128 the next S (or dP) goes over
the columns from which dV (or dK, dQ) takes its A operand, so the issuer must know by then that it is done: from a
commit issued behind it, or from a barrier of the compute warps, which arrive behind a commit of S or dP."""
import re

import pytest

from test_early_start import source

TOKEN = re.compile(r"(issue_s|issue_dp)\(j \+ 1\)|(?:mma_ts|slice)\((t_dq|t_dv|t_dk),|(commit)\((k\w+)|(wait)\(([^,]*)")
COMPUTE = {"kSFree": "kSFull", "kPHalf": "kSFull", "kPFull": "kSFull", "kDsFull": "kDpFull"}      # and the commit their arrivals are behind


def issued(name):
    """The issuer's step as (what, barrier or product); a product of S or dP with the waits in front of it."""
    text = source("attn_bwd.cu")
    body = text[text.index("void %s<D>::run(" % name):]
    step = body[body.index("issue_s(0)"):body.index("commit(kDone)")]
    for m in TOKEN.finditer(step):
        issue, product, commit, bar, wait, bars = m.groups()
        if issue:
            own = body[body.index("auto %s = " % issue):]
            for w in re.findall(r"wait\(([^,]*)", own[:own.index("mma_")]):
                yield "wait", re.findall(r"k[A-Z]\w+", w)[0]
            yield "issue", issue
        elif product:
            yield "product", product
        elif commit:
            yield "commit", bar
        else:
            yield "wait", re.findall(r"k[A-Z]\w+", bars)[0]


@pytest.mark.parametrize("name,overwrites", [("DqBlock", {"issue_dp": {"t_dq"}}),
                                             ("DkdvBlock", {"issue_s": {"t_dv"}, "issue_dp": {"t_dk"}})])
def test_operands_are_read_before_they_are_overwritten(name, overwrites):
    pending, covers, checked = set(), {"kSFull": set(), "kDpFull": set()}, []
    for what, x in issued(name):
        if what == "product":
            pending.add(x)
            for c in covers.values():
                c.discard(x)
        elif what == "commit":
            covers[x] = set(pending)                   # a commit is behind everything issued before it
        elif what == "wait":
            pending -= covers.get(COMPUTE.get(x, x), set())
        else:
            assert not pending & overwrites.get(x, set()), "%s over the operand of a product that may still run" % x
            checked.append(x)
            covers["kSFull" if x == "issue_s" else "kDpFull"] = set(pending)
    assert checked == ["issue_s", "issue_dp"]

"""The order in which the GRU recurrence reuses its staging buffers, checked on
the host: a model of who waits for whom in a round (csrc/gru_common.cuh,
push_rows_bulk), with the number of buffers that the kernels are built with."""
import functools
import os
import re

import pytest

from paper_1810_09958_gb300 import build, isam

SMS, SMEM = 152, 232448


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    isam.load()


def staging_buffers():
    with open(os.path.join(build.CSRC, "gru_common.cuh")) as f:
        m = re.search(r"constexpr int kGruStages = (\d+);", f.read())
    return int(m.group(1)) if m else 1


def copies_land_before(H, reset_before, buffers):
    """Whether every copy out of a staging buffer has landed before the buffer is
    written again.  CTA c of the hidden size's groups of 32 units; a round's events:
    gather (needs the vectors that its K range's CTAs published), send (after its
    gather and its last reduction), land at each owner of its cluster, reduce
    (every row of the cluster has landed), publish the next round's vectors."""
    p = isam.gru_plan(1, 32, H, reset_before, num_sms=SMS, smem_optin=SMEM)
    ks, ka, n = p["splits"], p["atoms"], p["ctas"]
    uo = 32 // ks  # units whose gates one CTA evaluates
    cluster = lambda c: [c // ks * ks + r for r in range(ks)]
    reads = [sorted({u // uo for u in range(c % ks * ka * 64, min(H, (c % ks + 1) * ka * 64))}) for c in range(n)]

    @functools.cache
    def landed(kind, c, k):
        """Copies (from, round) out of CTA 0's cluster known to have landed at all owners when the event happens."""
        if k < 0:
            return frozenset()
        if kind == "publish":  # round k's vectors
            return landed("reduce", c, k - 1)
        if kind == "send":
            return frozenset().union(landed("reduce", c, k - 1), *(landed("publish", q, k) for q in reads[c]))
        seen = frozenset().union(*(landed("send", q, k) for q in cluster(c)))
        return seen | {(q, c, k) for q in cluster(c) if q != c}

    step = 2 if reset_before else 1  # a gate's rows go out every step-th round
    k = 4
    for c in cluster(0):
        again = next(r for r in range(k + step, k + 9, step) if r % buffers == k % buffers)
        if not {(c, o, k) for o in cluster(0) if o != c} <= landed("send", c, again):
            return False
    return True


@pytest.mark.parametrize("reset_before", [False, True])
def test_staged_rows_have_landed_before_their_buffer_is_written_again(reset_before):
    for H in range(64, 1025, 96):  # 1, 2 and 4 splits, even and uneven K ranges
        if isam.gru_plan(1, 32, H, num_sms=SMS, smem_optin=SMEM)["splits"] > 1:
            assert copies_land_before(H, reset_before, staging_buffers()), H


def test_one_staging_buffer_would_not_be_enough():
    """The model sees the difference: with one buffer the next round's writes come
    too early unless the reset gate's second round lies in between."""
    assert not copies_land_before(1024, False, 1)
    assert copies_land_before(1024, True, 1)

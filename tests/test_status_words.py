"""Status words that other CTAs write: the threads of a CTA must not decide on them one by one.

A thread that leaves (or takes another way) because of a status word that the thread beside it
read a moment earlier leaves that one at a named barrier, which has no limit.  So every `if` on
such a word is a vote of the CTA (bar_named_or, __syncthreads_or), the choice of one thread for
all, or a poll inside a bounded wait whose outcome the CTA shares.
"""
import glob
import os

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1805_01559_gb300", "csrc")
VOTE = ("bar_named_or(", "__syncthreads_or(")
ONE_THREAD = ("tid == 0", "threadIdx.x == 0")
POLL = ("(n & 63)", "(++n & 1023)")
# written two grid barriers before it is read, and again only after the next one
STABLE = ("&P.st->absorb[s & 1]",)


def test_status_words_are_read_for_the_whole_cta():
    bad = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for n, line in enumerate(open(path), 1):
            if "if (" not in line or "ld_volatile_i32(" not in line:
                continue
            if os.path.basename(path) == "ot_common.cuh" and "ok = 0; break;" in line:
                continue  # thread 0's poll in grid_barrier
            if not any(k in line for k in VOTE + ONE_THREAD + POLL + STABLE):
                bad.append(f"{os.path.basename(path)}:{n}: {line.strip()}")
    assert not bad, "\n".join(bad)

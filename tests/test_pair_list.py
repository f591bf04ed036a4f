"""The bound of the shift's list of (source, neighbour) pairs, on the CPU: a
mixed cell has up to 26 pairs and a grid up to 2^31 - 1 cells, so the pairs
outnumber what a 32-bit counter holds.  The append of csrc/vof_shift.cu is read
from the source and run in small words."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2001_03477_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as fh:
        return re.sub(r"//[^\n]*", "", fh.read())


def test_append_is_unsigned_and_stops_at_a_full_list():
    text = source("vof_shift.cu")
    assert re.search(r"if \([^)]*\broom\b[^{]*\{\s*const unsigned k = atomicAdd\(sc\.npairs, 1u\);\s*"
                     r"room = k < sc\.pair_cap;\s*if \(room\) sc\.pairs\[k\] =", text)
    assert len(re.findall(r"npairs, 1", text)) == 1
    header = source("vof_launch.h")
    assert len(re.findall(r"unsigned pair_cap;", header)) == 2 and "unsigned* npairs;" in header
    assert not re.search(r"\bint pair_cap|\bint\* npairs", header)
    # the reader compares the same unsigned count
    assert re.search(r"const unsigned np = \(unsigned\)A\.cnt\[2\];", text)
    assert re.search(r"const bool listed = np <= A\.pair_cap;", text)


def test_count_stays_bounded():
    """The rule in 8-bit words: cap 2^7 - 1 (the largest N), 100 threads that each
    offer 26 pairs of many cells.  No index reaches the cap, the counter does
    not come round, and a full list is seen as such."""
    cap, threads, offers = 127, 100, 26 * 40
    count, stored = 0, []
    room = [True] * threads
    for _ in range(offers):  # every thread offers a pair
        for t in range(threads):
            if room[t]:
                k, count = count, count + 1
                assert count < 256  # no wrap
                room[t] = k < cap
                if room[t]:
                    stored.append(k)
    assert sorted(stored) == list(range(cap)) and count > cap
    # the kernel's own numbers: 152 x 4 CTAs of 128 threads, N < 2^31
    text = source("vof_shift.cu")
    ctas, thr = re.search(r"kListCTAs = 152 \* (\d+);", text), re.search(r"kListThreads = (\d+);", text)
    assert 2 ** 31 - 1 + 152 * int(ctas.group(1)) * int(thr.group(1)) < 2 ** 32

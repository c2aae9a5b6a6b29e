"""The grid barrier's word: a release and an acquire synchronise only if they access the same bytes, so
every access to it in the device code has one width."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1311_7477_gb300", "csrc")


def test_barrier_accesses_have_one_width():
    src = open(os.path.join(CSRC, "dg_device.cuh")).read()
    body = re.search(r"bool grid_barrier\(.*?\n}\n", src, re.S).group(0)
    asm = re.findall(r'asm volatile\("(\S+) [^"]*"[^;]*"l"\((&?s(?:->\w+)?)\)', body)
    ops = [op for op, _ in asm]
    assert {op.split(".")[0] for op in ops} == {"ld", "red"}
    assert {op[-3:] for op, _ in asm} == {"u64"}
    assert len({place for _, place in asm}) == 1
    word = asm[0][1].split("->")[1]
    assert re.search(r"unsigned long long %s;" % word, src)
    # nothing else of the barrier touches the word or a part of it, but the whole-word error
    assert re.findall(r"atomic\w+\(([^,]*), \(([\w ]+)\)", body) == [("&s->" + word, "unsigned long long")]
    # long waits poll without an acquire (it drops the L1 lines of the blocks still at work on the SM) and
    # acquire once they have seen the last arrival
    assert [op.split(".")[1] for op in ops] == ["release", "acquire", "relaxed", "acquire"]
    assert re.search(r"if \(spins >= kAcquirePolls\)\s*asm volatile\(\"ld.acquire", body)

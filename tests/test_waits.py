"""The softmax threads of the tcgen05 attention wait several times a tile.  An expired wait must not be overwritten by a later one, which
may find its barrier complete in the meantime: a part of a row would be missing and no error word up.  (Read off the source: an
expired wait is nothing to cause on a GPU.)"""
import os
import re

from paper_2510_04147_b200 import build


def test_the_softmax_threads_forget_no_expired_wait():
    with open(os.path.join(build.CSRC, "attention_verify_pipe.cu")) as f:
        source = f.read()
    loop = source[source.index("softmax threads (log2 domain)"):source.index("this CTA's last part;")]
    waits = re.findall(r"(.*)\bmbar_wait\(", loop)
    assert len(waits) >= 4 and all(w.strip() == "ok = ok &&" for w in waits), waits
    for word in re.findall(r"\bok = (?!ok && mbar_wait)([^;]*);", loop):       # what else sets it keeps what it was
        assert re.fullmatch(r"softmax_barrier_and\(ok\)|__all_sync\(0xffffffffu, ok \? 1 : 0\) != 0", word), word

"""The tensor-core pass's diagnostic counters: one name each in the binding, and
each added to somewhere in the kernel."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def read(*path):
    with open(os.path.join(ROOT, "paper_1304_4327_gb300", *path)) as f:
        return f.read()


def test_every_counter_is_named_and_fed():
    src = read("csrc", "knn_tc.cuh")
    counters = re.findall(r"\bTT_\w+", src[src.index("enum TcTimer {"):src.index("static_assert(TT_N")].split("TT_N")[0])
    counters = list(dict.fromkeys(counters))
    names = re.search(r"TC_TIMERS = \((.*?)\)", read("dtree.py"), re.S).group(1)
    assert len(re.findall(r'"\w+"', names)) == len(counters)
    uses = src[src.index("static_assert(TT_N"):] + src[:src.index("enum TcTimer {")]
    fed = set(re.findall(r"timers\[(TT_\w+)\]", uses)) | set(re.findall(r"&x\.timers\[[^\]]*?(TT_\w+)", uses))
    assert not [c for c in counters if c not in fed]

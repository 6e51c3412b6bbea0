"""There is one bounded mbarrier wait in the sources, and its self-test runs the one that the tensor-core stage uses."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1804_02718_gb300", "csrc")


def test_the_selftest_runs_the_wait_that_is_used():
    src = {n: re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, n)).read()) for n in os.listdir(CSRC)}
    where = [n for n, s in src.items() for _ in re.findall(r"mbarrier\.try_wait", s)]
    assert where == ["dft16_tc.cu"], where
    s = src["dft16_tc.cu"]
    name = re.findall(r"bool (\w+)\(uint32_t \w+, uint32_t \w+\) \{\s*for[^}]*mbarrier\.try_wait", s, flags=re.S)[0]
    for kernel in ("k_dft16_tc", "k_wait_selftest"):
        body = s[s.index(kernel + "("):].split("\n}\n")[0]
        assert re.search(r"\b%s\(" % name, body), kernel

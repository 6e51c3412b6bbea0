"""No stream or event is used whose creation was not checked: work on a null stream would run outside the graph that is being
captured.  (A failing creation cannot be had on purpose; the check is in the source.)"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1804_02718_gb300", "csrc")


def test_stream_and_event_creation_is_checked():
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            for i, line in enumerate(f, 1):
                assert not re.match(r"\s*cuda(Stream|Event)Create", line), (name, i, line)

"""The library keeps no state of its own behind its contexts: what a context asks of its device it keeps itself, so that
contexts of several threads and devices do not share it. The static estimate's scratch, made once per device under a lock,
is the exception that the header describes."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1402_0266_gb300", "csrc")
STATE = re.compile(r"^\s+(?:static|thread_local)\s+(?!const\b|constexpr\b|void\b|_assert)[\w:<>*& ]+?\w+(?:\[[^\]]*\])*\s*(?:=|;|\{)", re.M)


def test_functions_hold_no_static_variables():
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        found = STATE.findall(text)
        assert not found, (name, found)

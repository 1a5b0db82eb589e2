"""Every bounded device-side wait of the library is one of two functions (wait_arrivals,
mbar_wait), and the test entry of the timeout path (mor_debug_wait_timeout) runs the
exchange that the reduced solve runs, so that what it shows holds for the solve.  Read from
the sources: the waits of a healthy solve never run out."""
import glob
import os
import re

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2404_06260_gb300", "csrc")


def _sources():
    out = {}
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        out[os.path.basename(path)] = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(),
                                             flags=re.S)
    return out


def _function(text, name):
    at = re.search(r"\b%s\([^;{]*\)\s*\{" % name, text)
    depth, k = 1, at.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        k += 1
    return text[at.start():k]


def test_clock_budgets_only_in_the_two_wait_functions():
    left = {}
    for name, text in _sources().items():
        for fn in ("wait_arrivals", "mbar_wait"):
            if re.search(r"\b%s\([^;{]*\)\s*\{" % fn, text):
                text = text.replace(_function(text, fn), "")
        if "clock64" in text or "globaltimer" in text:
            left[name] = text.count("clock64")
    assert not left


def test_the_timeout_entry_runs_the_solve_s_exchange():
    text = _sources()["mor_reduced.cu"]
    exchange = _function(text, "rcg_exchange")
    assert "wait_arrivals(" in exchange
    assert "rcg_exchange(" in _function(text, "k_rcg_grid")
    api = _function(_sources()["mor_api.cu"], "mor_debug_wait_timeout")
    launch = re.search(r"\b(launch_\w+)\(", api).group(1)
    kernel = re.search(r"\b(k_\w+)\s*<<<", _function(text, launch)).group(1)
    assert "rcg_exchange(" in _function(text, kernel)

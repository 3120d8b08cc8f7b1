"""Every entry point of qis_api.cu that launches kernels makes the context's device current first (a launch
into a stream of another device fails): on a new host thread, or after work on another context, the
current device can be any."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2010_00180_gb300", "csrc", "qis_api.cu")
LAUNCHES = r"\bLAUNCH\(|\bbuild_work\(|\blaunch_iteration\w*\(|\bimport_search\(|\bmlp_propose_states\("


def entry_points():
    """(name, body) of the functions of the library's C interface, and of flush_init, which many call first."""
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    for m in re.finditer(r"^(?:int|void|const char\*) (qis_\w+|flush_init)\([^;{]*\) \{\n(.*?)^\}", text, re.M | re.S):
        yield m.group(1), m.group(2)


def test_device_is_set_before_the_first_launch():
    seen = 0
    for name, body in entry_points():
        m = re.search(LAUNCHES, body)
        if not m:
            continue
        seen += 1
        assert "cudaSetDevice(" in body[: m.start()], name
    assert seen >= 10

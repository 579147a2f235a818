"""kt_network_load parses and packs tables only: the programs of the group and team kernels are
laid out by the first call that integrates, under the network's lock (csrc/kt_api.cu)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_04941_gb300", "csrc")


def _body(code, head):
    part = code[code.index(head):]
    return part[:part.index("\n}\n")]


def test_load_lays_out_no_programs():
    with open(os.path.join(CSRC, "kt_api.cu")) as f:
        code = re.sub(r"//[^\n]*", "", f.read())
    callers = [m.start() for m in re.finditer(r"\bbuild_(?:coop|team)\((?!kt_network)", code)]
    lay = code.index("int kt_network::lay_out()")
    assert callers and all(lay < at < lay + len(_body(code, "int kt_network::lay_out()")) for at in callers)
    for entry in ("int kt_network_load(", "int kt::network_element_basis("):
        assert "lay_out" not in _body(code, entry) and "device_blob" not in _body(code, entry)

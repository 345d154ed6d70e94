"""Uploads are ordered with the kernels that read them: every host-to-device
copy and every fill of the library goes to the context's own stream.  A plain
cudaMemcpy or cudaMemset works on the legacy default stream, which a
non-blocking stream (PyTorch's side streams) does not wait for."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_1511_04519_gb300" / "csrc"


def _calls(name):
    for f in sorted(CSRC.glob("*")):
        text = f.read_text()
        for m in re.finditer(r"\b%s\(" % name, text):
            depth, i = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(text[i], 0)
                i += 1
            yield f.name, text[m.start():i]


def test_no_upload_or_fill_on_the_default_stream():
    assert not [c for c in _calls("cudaMemcpy") if "DeviceToHost" not in c[1]]
    assert not list(_calls("cudaMemset"))


def test_asynchronous_copies_name_a_stream():
    calls = list(_calls("cudaMemcpyAsync"))
    assert calls
    for f, c in calls:
        assert re.search(r"(\bst|->st)\)$", c), (f, c)

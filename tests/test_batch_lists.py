"""The batch's work lists and the captured step that holds their addresses, on the source: a
replay on freed lists cannot be staged on a GPU that others share."""
import os
import re

SRC = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                        "paper_1409_5474_gb300", "csrc", "batch.cu")).read()
SRC = re.sub(r"//[^\n]*", "", SRC)


def _body(name):
    return re.search(r"\n[\w\s]*\b%s\([^;{}]*\)\n\{(.*?)\n\}" % name, SRC, flags=re.S).group(1)


def test_the_captured_step_goes_before_the_lists():
    body = _body("build_items")
    drop = body.index("drop_graph(b);")
    assert all(drop < m.start() for m in re.finditer(r"cudaFree\(b->d_(items|groups|part)\)", body))
    # and the counts say that there are no lists until both are uploaded
    assert drop < body.index("b->nitems = b->ngroups = 0;") < body.index("cudaFree(")
    last = max(m.end() for m in re.finditer(r"BCK\(", body))
    assert body.index("b->nitems = (int)items.size();") > last
    assert body.index("b->ngroups = (int)groups.size();") > last


def test_no_step_is_taken_without_lists():
    for name in ("launch_batch_force", "capture_step"):
        body = _body(name)
        assert 0 <= body.index("ensure_items(b)") < body.index("batch_force(b)")
    # the lists are used nowhere else
    assert len(re.findall(r"\bbatch_force\(b\)", SRC)) == 2

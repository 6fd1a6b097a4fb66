"""Kernels that may start before the one before them in the stream has ended read
nothing of its results before they have waited for it, or have taken the draw list
over by an acquire (k_raster_fast). Checked in the source of the kernels."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = os.path.join(ROOT, "paper_2204_01287_gb300", "csrc", "raster.cu")

# what reads or writes memory that a kernel of the stream writes
TOUCHES = re.compile(r"entry_counts\(|clear_view\(|publish_frame\(|take_list\(|next_entry\(|flush_atomics\(|"
                     r"\bs\.(entries|counters|acc|stats|lod_sel)\b|\bc\.(batches|w1|w2|w3|color|parent)\b|\.vis\b")


def _text():
    with open(SOURCE) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _body(text, name):
    """The braces' text of the function `name`."""
    at = re.search(r"\b" + name + r"\([^;{]*\)\s*\{", text).end()
    depth, i = 1, at
    while depth:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
    return text[at:i]


def test_early_kernels_wait_before_they_read():
    text = _text()
    kernels = set(re.findall(r"launch_early\((k_\w+)", text))
    assert {"k_begin", "k_raster_fast", "k_raster_general", "k_raster2", "k_rasterN", "k_resolve"} <= kernels
    for k in sorted(kernels):
        body = _body(text, k)
        first = TOUCHES.search(body)
        wait = body.find("wait_for_previous();")
        assert wait >= 0, k
        assert wait < first.start() or first.group() == "take_list(", (k, first.group())


def test_the_list_is_taken_over_by_release_and_acquire():
    text = _text()
    take, give = _body(text, "take_list"), _body(text, "give_list")
    assert "ld.acquire.gpu" in take and "st.release.gpu" in give
    # without this frame's number: the wait, then the counters
    assert 0 < take.find("ld.acquire.gpu") < take.find("!= s.frame") < take.find("wait_for_previous();") \
        < take.find("entry_counts(")
    general = _body(text, "k_raster_general")
    assert general.find("wait_for_previous();") < general.find("give_list(") < general.find("start_next();")

"""What the library prepares outside a caller's stream is there before any
stream can use it.

Work on the legacy default stream is not ordered before work on a non-blocking
stream (PyTorch's streams are such), cudaMemset returns before it has run, and
a copy from pageable memory may return before it has arrived.  A missing wait
shows on a GPU only by chance, so the sources are checked: fills go through
zero_now, which waits, and whatever copies a batch's tables or a volume's nodes
waits after the last copy.  A batch's tables are rewritten only once no step
that reads them is in flight."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_24236_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def body(text, head):
    """The function whose definition contains `head`, up to its closing brace."""
    at = text.index(head)
    return text[at:text.index("\n}", at)]


def test_fills_outside_a_callers_stream_are_waited_for():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        assert "cudaMemset(" not in source(os.path.basename(path)), path
    fill = body(source("pf_internal.cuh"), "zero_now(void* p")
    assert 0 < fill.index("cudaMemsetAsync(p, 0, bytes, z)") < fill.index("cudaStreamSynchronize(z)")


def test_host_copies_are_waited_for():
    for name, head in (("track.cu", "pf_status batch_tables("), ("volume.cu", "pf_status pf_volume_upload_impl(")):
        text = body(source(name), head)
        last = text.rindex("cudaMemcpyHostToDevice")
        assert re.search(r"cuda(Device|Stream)Synchronize\(", text[last:]), name
    create = body(source("track.cu"), "pf_status pf_batch_create(")
    assert create.rindex("cudaMemcpyHostToDevice") < create.index("batch_tables(b, false)")  # which waits


def test_batch_tables_are_rewritten_between_steps():
    tables = body(source("track.cu"), "pf_status batch_tables(")
    assert tables.index("cudaDeviceSynchronize()") < tables.index("cudaMemcpyHostToDevice")
    # every change of a table goes through there
    assert source("track.cu").count("cudaMemcpy(b->d_args") == 1

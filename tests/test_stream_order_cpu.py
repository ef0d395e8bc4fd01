"""Every copy and fill that a kernel on a caller's or a non-blocking stream reads is
queued on that stream: a plain cudaMemcpy from pageable memory returns once the data is
staged, and cudaMemset before it has run, so that nothing orders another stream after
them.  Read from the source: on a GPU a lost race shows as a write out of range."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1507_00895_gb300", "csrc")


def legacy_stream_calls(name):
    txt = open(os.path.join(CSRC, name)).read()
    txt = re.sub(r"//[^\n]*|/\*.*?\*/", "", txt, flags=re.S)
    return re.findall(r"\bcuda(?:Memcpy|Memset)\s*\([^;]*;", txt)


def test_batch_tables_go_up_on_the_batch_stream():
    assert legacy_stream_calls("df_batch.cu") == []


def test_network_and_handle_set_up_on_their_own_streams():
    assert legacy_stream_calls("df_mlp.cu") == []
    # (df_selftest_wait launches on the legacy stream itself)
    calls = [c for c in legacy_stream_calls("df_api.cu") if not re.match(r"cudaMem(set|cpy)\((d, 0|&h, d),", c)]
    assert calls == []

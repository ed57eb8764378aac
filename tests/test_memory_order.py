"""What memory the kernels touch and in which order, where no run shows it reliably: looked up in their source. CPU only."""
import os
import re

import pytest

from conftest import ROOT


def body(file, head):
    """The brace-matched body, without comments, of the first function whose declaration contains `head`."""
    text = re.sub(r"//.*", "", open(os.path.join(ROOT, "paper_2009_13003_b200", "csrc", file)).read())
    begin = text.index("{", text.index(head))
    depth = 0
    for i in range(begin, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[begin: i + 1]
    raise AssertionError(head)


def test_a_rejected_stream_is_reported_behind_the_launch_before():
    # The launch before a chain's later one may be the one that clears the status word: an error set ahead of
    # wait_previous() could be cleared again. Only that clearing itself, in the first launch, is ahead of it.
    text = body("lc_decode.cu", "void decode_vector(")
    ahead = text[: text.index("wait_previous()")]
    assert re.findall(r"status\s*\.\s*\w+[^;]*;", ahead) == ["status.word = 0;"]
    assert "status.set(err)" in text[len(ahead):]


def test_the_last_warp_to_arrive_reads_the_sizes_behind_a_fence():
    # Every warp writes its chunk's size, then (behind a fence) adds itself to the count; lane 0 of the last one sees the
    # count, other lanes read the sizes.
    text = body("lc_encode.cu", "encode_kernel(Control*")
    write, count = text.index("s_chunk_bytes[buf][warp] = chunk_bytes"), text.index("atomicAdd(&s_arrived[buf]")
    read = text.index("&s_chunk_bytes[buf][lane]")
    assert write < text.index("__threadfence_block()", write) < count
    branch = text[text.index("arrival == kEncWarps - 1", count): read]
    assert 0 < branch.find("__threadfence_block()") < branch.find("__syncwarp()")


@pytest.mark.parametrize("file,head", [("lc_encode.cu", "encode_kernel(Control*"), ("lc_encode.cu", "encode_sizes_kernel(const Control*"),
                                       ("lc_segments.cu", "segments_encode_kernel(Control*")])
def test_only_kernels_with_code_tables_send_the_slow_path_to_them(file, head):
    # The tables lie at the start of the dynamic shared memory, of which encode_sizes_kernel is launched with none.
    text = body(file, head)
    assert set(re.findall(r"\bchunk_slow(\S*?)\(", text)) == {"<true>" if "shared_tables()" in text else "<false>"}

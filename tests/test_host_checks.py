"""What the library decides on the host before it touches a device (made-up addresses, no GPU)."""
from paper_2009_13003_b200 import binding


def test_wait_checks_its_arguments():
    L, info = binding.lib(), binding.LCInfo()
    ws, stream, page = 0x40000, 0x30000, 0x50000
    assert L.lc_wait(None, stream, info, page, None) == binding.ERR_ARG
    assert L.lc_wait(ws + 16, stream, info, page, None) == binding.ERR_ARG
    assert L.lc_wait(ws, stream + 4, info, page, None) == binding.ERR_ARG
    assert L.lc_wait(ws, stream, None, page, None) == binding.ERR_ARG
    assert L.lc_wait(ws, stream, info, page + 8, None) == binding.ERR_ARG

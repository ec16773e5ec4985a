"""Device bytes of a batch's argument records: nothing where they go as kernel parameters (up to 36
members), otherwise at most one 416-byte (FP64: 480-byte) record per phase and member with the block
prefix and the period count, so that a server's fixed arena keeps its room for lattices."""
import pytest

from paper_2403_15768_gb300 import klb


@pytest.mark.parametrize("storage,record,phases", [("fp64", 480, 6), ("fp32", 416, 6), ("fp16", 416, 384), ("bf16", 416, 384)])
@pytest.mark.parametrize("n", [1, 8, 36, 37, 64, 400])
def test_table_bytes(storage, record, phases, n):
    bytes_ = klb.klb_server_table_bytes(klb.STORAGE[storage], n)
    most = 256 if n <= 36 else phases * n * record + 4 * (n + 1) + 3 * 256
    assert 0 < bytes_ <= most

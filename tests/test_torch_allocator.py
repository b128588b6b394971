"""The allocator that the binding hands to the library takes blocks on the stream that the library names
(CPU: torch's caching allocator is replaced)."""
import torch

from paper_2308_00106_gb300 import maxe


def test_blocks_are_taken_on_the_named_stream(monkeypatch):
    asked, freed = [], []

    def alloc(size, device=None, stream=None):
        asked.append((size, stream))
        return 0x1000 * len(asked)

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", alloc)
    monkeypatch.setattr(torch.cuda, "caching_allocator_delete", freed.append)
    for nbytes, stream in ((1000, 0x7F00), (1, None), (0, 0x7F08)):
        p = maxe._ALLOC.alloc(nbytes, None, stream)
        assert p == 0x1000 * len(asked)
        maxe._ALLOC.free(p, None, stream)
    assert asked == [(1000, 0x7F00), (1, 0), (1, 0x7F08)]  # no stream: the default stream
    assert freed == [0x1000, 0x2000, 0x3000]


def test_out_of_memory_is_a_null_block(monkeypatch):
    def alloc(size, device=None, stream=None):
        raise torch.cuda.OutOfMemoryError("none left")

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", alloc)
    assert maxe._ALLOC.alloc(1 << 40, None, None) is None
    maxe._ALLOC.free(None, None, None)

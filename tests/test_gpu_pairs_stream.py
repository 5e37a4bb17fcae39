"""vx_radix_sort_pairs in a context over a caller's arena and stream: work that
the caller has given the stream before the call still sees the arena's old
contents, whichever streams the call itself uses, and the sort is right."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

vx = pytest.importorskip("paper_2502_09541_gb300")
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [1000, 32_767, 32_768, 1_000_003])
def test_work_queued_before_the_call_reads_the_arena_first(n):
    rng = np.random.default_rng(n)
    k = rng.integers(0, 2**64 - 1, n, dtype=np.uint64)
    v = np.arange(n, dtype=np.uint32)
    arena = torch.arange(16 << 20, dtype=torch.int32, device="cuda")
    seen = torch.zeros_like(arena)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    c = vx.vx_open_ex(arena.data_ptr(), arena.numel() * 4, stream.cuda_stream)
    try:
        with torch.cuda.stream(stream):
            torch.cuda._sleep(100_000_000)  # about 50 ms
            seen.copy_(arena)
        ok, ov = vx.vx_radix_sort_pairs(c, k, v)
        torch.cuda.synchronize()
    finally:
        vx.vx_close(c)
    assert torch.equal(seen, torch.arange(16 << 20, dtype=torch.int32, device="cuda"))
    perm = np.argsort(k, kind="stable")
    assert np.array_equal(ok, k[perm]) and np.array_equal(ov, v[perm])

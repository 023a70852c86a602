"""The autotuners time their sort candidates on the radix sort, whose launch shapes they
choose, not on builds by bins, which have one shape: the times are those of the longer
way, and the digit widths differ by more than noise."""
import ctypes

import pytest

torch = pytest.importorskip("torch")

from paper_2110_11616_gb300 import cga

pytestmark = pytest.mark.gpu
BITS, N = 12, 12_000_000


def _points(n, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.rand((n, 3), generator=gen, device="cuda")


@pytest.fixture()
def clean():
    def clear():
        for bits in range(1, 17):
            for nb in range(32):
                cga.tuning_set(bits, (1 << (nb - 1)) if nb else 0, None)

    clear()
    yield
    clear()


def _least_ms(call):
    call()
    best = float("inf")
    for _ in range(5):
        t0, t1 = torch.cuda.Event(True), torch.cuda.Event(True)
        torch.cuda.synchronize()
        t0.record()
        kept = call()
        t1.record()
        torch.cuda.synchronize()
        best = min(best, t0.elapsed_time(t1))
        del kept
    return best


def test_cloud(clean):
    g, pts = cga.grid_from_box([0, 0, 0], 1.0, BITS), _points(N, 1)
    build = _least_ms(lambda: cga.cga_build(pts, g))
    _, times = cga.cga_autotune(pts, g)
    sort = list(times["sort"].values())
    assert min(sort) > 1.3 * build, (build, times)   # 2.0 at this size
    assert max(sort) > 1.03 * min(sort), times


def test_pipeline(clean):
    pts = [_points(N // 4, 2 + i) for i in range(2)]
    grids = [cga.grid_from_box([0, 0, 0], 1.0, BITS)] * 2
    xform = [[1.0, 0.0, 0.0, 0.0, 1.0, 0.0, 0.0, 0.0, 1.0, 0.01, 0.0, 0.0]] * 2
    pipe = cga.Pipeline(pts, grids, xform, [None] * 2)
    run = _least_ms(pipe.run_graph)
    _, times = cga.pipeline_autotune(pts, grids, xform, [None] * 2)
    assert min(times["sort"].values()) > 1.15 * run, (run, times)
    assert max(times["sort"].values()) > 1.02 * min(times["sort"].values()), times
    pipe.free()


def test_entry_left_unset_by_an_error(clean):
    """After a failed autotune a merge still takes its partition from the rule: the blocks
    that it asks for are those of before, and others once the default is set."""
    sizes, held = [], {}

    @ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p)
    def alloc(ctx, size, stream):
        sizes.append(int(size))
        t = torch.empty(int(size), dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = t
        return t.data_ptr()

    @ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p)
    def free(ctx, p, stream):
        torch.cuda.synchronize()
        held.pop(p, None)

    pts = _points(60_000, 9)
    g = cga.grid_from_box([0, 0, 0], 1.0, BITS)
    a, b = cga.cga_build(pts[0::2].contiguous(), g), cga.cga_build(pts[1::2].contiguous(), g)
    allocator = cga.Allocator(None, alloc, free)

    def merge_blocks():
        sizes.clear()
        m = cga.cga_merge(a, b, allocator=allocator)
        torch.cuda.synchronize()
        del m
        return list(sizes)

    before = merge_blocks()
    with pytest.raises(cga.CgaError):
        cga.cga_autotune(pts, cga.make_grid(BITS, float("nan"), (0.0, 0.0, 0.0)))
    assert merge_blocks() == before
    cga.tuning_set(BITS, len(pts), {"radix_bits": 8, "sort_threads": 512, "merge_half": 2048})
    assert merge_blocks() != before

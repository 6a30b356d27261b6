"""What the CUDA sources promise and no run can show: orderings whose absence
would only now and then give a wrong sum."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1112_0065_gb300", "csrc")


def _code(path):
    with open(path) as fh:
        return re.sub(r"//[^\n]*", "", fh.read())


def test_persistent_tiles_fence_before_the_next_tile():
    """A persistent CTA's tiles may have different shared-memory layouts, so
    that the copy engine writes where the tile before wrote with plain stores:
    after the tile routine every thread fences between the two, then the block
    meets."""
    loops = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        src = _code(path)
        for m in re.finditer(r"atomicAdd\(counter, 1ULL\)", src):
            loops.append(os.path.basename(path))
            rest = src[m.end():]
            tile = re.search(r"if \(!(?:gsum|dd)_tile<[^>]*>\([^;]*\)\) break;", rest)
            assert tile, path
            assert re.match(r"\s*tc::fence_async_smem\(\);\s*__syncthreads\(\);\s*}", rest[tile.end():]), path
    assert sorted(loops) == ["gsum.cu", "tiled_launch.cuh"]


def test_no_multiprocessor_count_in_the_code():
    """Grids and rules ask the device how many multiprocessors it has (the weight
    gradients' number of partial sums is fixed: it sets their order)."""
    for path in sorted(glob.glob(os.path.join(CSRC, "**", "*.cu*"), recursive=True)):
        assert not re.search(r"\b(152|304)\b", re.sub(r"kMaxPartials = 304", "", _code(path))), path


def test_tensor_maps_in_memory_are_fenced_by_the_threads_that_use_them():
    """Tensor maps that the host copied to global memory: the acquiring fence has
    system scope and is the issuing thread's own (lane 0 of each warp)."""
    assert "fence.proxy.tensormap::generic.acquire.sys" in _code(os.path.join(CSRC, "tma.cuh"))
    kernel = _code(os.path.join(CSRC, "gsum.cu")).split("dd_gsum_batch_kernel(")[1]
    assert re.search(r"if \(\(threadIdx\.x & 31\) == 0\)\s*for \(int b = 0; b < desc->nbeams; \+\+b\) "
                     r"tc::fence_tensormap\(&desc->map\[b\]\);", kernel)

"""Source checks of what no run can show: a hand-over that a warp acquires through one lane is ordered for its other lanes, no
warp waits without a limit for warps that may have given up, and shared memory that is read in 16-byte pieces is declared so."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_12932_b200", "csrc")


def code(name):
    """A source file without its // comments."""
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_one_lane_acquires_go_through_the_warp_form():
    """`lane == 0` polling with acquire orders memory for that lane alone: every kernel takes the form that ends in __syncwarp,
    and that form does."""
    for name in sorted(os.listdir(CSRC)):
        if name.endswith(".cu"):
            assert not re.search(r"(?<!warp_)wait_bit_acquire_gpu\(", code(name)), name
    body = re.search(r"bool warp_wait_bit_acquire_gpu\([^)]*\) \{(.*?)\n\}", code("ptx_sm100.cuh"), re.S).group(1)
    assert body.index("__shfl_sync") < body.index("__syncwarp();") < body.index("return")


def test_no_barrier_inside_the_roles_of_the_tensor_core_kernels():
    """Their roles leave their loops one by one when a wait runs out, so a barrier among some warps could wait for good: the only
    block barriers are the two that every thread reaches, after the set-up and before tensor memory is given back."""
    for name in ("gemm_tcgen05.cu", "gemm_tcshort.cu"):
        text = code(name)
        assert "named_bar_sync" not in text and "bar.sync" not in text and text.count("__syncthreads()") == 2, name


def test_drain_warps_agree_ahead_of_tensor_memory_loads():
    """tcgen05.ld is executed by whole warps: lanes that saw different outcomes of a look at a barrier, or of a wait that runs
    out, must not part ways there.  The tall-tile kernel looks ahead, so each of its drain's looks and waits is the voting form."""
    text = code("gemm_tcgen05.cu")
    drain = text[text.index("setmaxnreg.inc"):text.index("bulk_wait_group0")]
    assert "ready" in drain and "tmem_ld_32x32" in drain
    assert not re.findall(r"(?<!warp_)mbar_(?:test_|try_)?wait\w*\(", drain)
    for form in ("warp_mbar_wait", "warp_mbar_wait_hot", "warp_mbar_test_wait"):
        body = re.search(r"bool " + form + r"\([^)]*\) \{(.*?)\n\}", code("ptx_sm100.cuh"), re.S).group(1)
        assert "__all_sync(0xFFFFFFFFu" in body, form


def test_waits_for_a_whole_tile_park():
    """The per-channel drain waits as long as a tile takes; polling for that time slows the unpack warps beside it."""
    assert re.findall(r"(\w*wait\w*)\(bar\(TILE_DONE", code("gemm_tcgen05.cu")) == ["warp_mbar_wait"]


def test_a_calls_number_is_read_once():
    """In the fused gate+up step's one-kernel form every further read of the number would be a round trip in the launch's tail."""
    text = code("gemm_strip.cu")
    text = text[text.index("gemm_strip_kernel("):text.index("requant_kernel(")]
    assert text.count("__ldcg(&a.sync->done)") == 1
    assert re.findall(r"sync->done ([^;]*);", text) == ["= call"]


def test_shared_tables_read_in_16_byte_pieces_are_aligned():
    """A float2 table is 8-byte aligned by its type; where the compiler places it today is no promise."""
    text = code("streaming.cu")
    names = re.findall(r"reinterpret_cast<const float4\*>\(&(\w+)\[", text)
    assert names
    for name in names:
        assert re.search(r"__shared__ (__align__\(16\) float2|float4) " + name + r"\[", text), name

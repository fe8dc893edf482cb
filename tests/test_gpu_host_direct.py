"""w4a8_linear_host with and without copies: pinned and pageable buffers, below and above the size up to which the kernels
read and write pinned memory themselves, every kernel family; the result is w4a8_linear's bit for bit."""
import numpy as np
import pytest
import torch

from paper_2608_12932_b200 import binding as B
from paper_2608_12932_b200 import workload as wl
from tests.gpu_util import DeviceLayer, bits, t_u16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N", [(1, 256, 256), (8, 4096, 6144), (16, 1024, 384), (12, 1024, 6144), (40, 1024, 512), (300, 1024, 512)])
@pytest.mark.parametrize("pin_x,pin_y", [(True, True), (True, False), (False, True), (False, False)])
def test_equals_the_device_path(M, K, N, pin_x, pin_y):
    case = wl.make_layer(K, N, 90 + M, M)
    layer = DeviceLayer(case, M)
    want = bits(B.w4a8_linear(t_u16(case["x"], torch.bfloat16), layer.packed, N, layer.ws))
    x = torch.from_numpy(case["x"].view(np.int16)).view(torch.bfloat16)
    y = torch.full((M, N), float("nan"), dtype=torch.bfloat16)
    x, y = x.pin_memory() if pin_x else x, y.pin_memory() if pin_y else y
    linear = B.HostLinear(M, N, K, layer.packed, layer.ws)
    for _ in range(2):
        linear(x, y)
        torch.cuda.synchronize()
        assert np.array_equal(y.view(torch.int16).numpy().view(np.uint16), want)
        y.fill_(float("nan"))


@pytest.mark.parametrize("M,K,N", [(1, 256, 256), (8, 4096, 6144), (16, 1024, 384), (12, 1024, 6144), (40, 1024, 512), (3, 16384, 128)])
def test_new_inputs_in_the_same_buffers_and_the_device_copies(M, K, N):
    """Every call reads what the pinned buffer holds at that time, and leaves x and y in the device staging buffers too."""
    case = wl.make_layer(K, N, 90 + M, 3 * M)
    layer = DeviceLayer(case, M)
    linear = B.HostLinear(M, N, K, layer.packed, layer.ws)
    linear.x_dev.fill_(7.0), linear.y_dev.fill_(7.0)
    x = torch.empty((M, K), dtype=torch.bfloat16).pin_memory()
    y = torch.empty((M, N), dtype=torch.bfloat16).pin_memory()
    for i in range(3):
        x_bits = case["x"][i * M:(i + 1) * M]
        want = bits(B.w4a8_linear(t_u16(x_bits, torch.bfloat16), layer.packed, N, layer.ws))
        x.view(torch.int16).copy_(torch.from_numpy(x_bits.view(np.int16)))
        linear(x, y)
        torch.cuda.synchronize()
        assert np.array_equal(y.view(torch.int16).numpy().view(np.uint16), want)
        assert np.array_equal(bits(linear.x_dev), x_bits) and np.array_equal(bits(linear.y_dev), want)


@pytest.mark.parametrize("M,K,N", [(8, 1024, 6144), (40, 1024, 512)])
def test_captured_into_a_graph(M, K, N):
    """The questions to the driver about the host buffers are asked at capture; a replay reads what the buffer holds then."""
    case = wl.make_layer(K, N, 95 + M, 2 * M)
    layer = DeviceLayer(case, M)
    linear = B.HostLinear(M, N, K, layer.packed, layer.ws)
    x = torch.zeros((M, K), dtype=torch.bfloat16).pin_memory()
    y = torch.empty((M, N), dtype=torch.bfloat16).pin_memory()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        linear(x, y)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        linear(x, y)
    for i in range(2):
        x_bits = case["x"][i * M:(i + 1) * M]
        want = bits(B.w4a8_linear(t_u16(x_bits, torch.bfloat16), layer.packed, N, layer.ws))
        x.view(torch.int16).copy_(torch.from_numpy(x_bits.view(np.int16)))
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(y.view(torch.int16).numpy().view(np.uint16), want)
        assert np.array_equal(bits(linear.x_dev), x_bits) and np.array_equal(bits(linear.y_dev), want)

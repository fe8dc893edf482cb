"""The per-token maxima that the fused gate+up call keeps in the workspace between its projection and its requantisation are never
cleared: each call's supersede the last call's.  So a workspace that has served calls with larger values, other token
counts and the other form gives the bits of a fresh one."""
import numpy as np
import pytest
import torch

from oracle import w4a8_oracle as onp
from paper_2608_12932_b200 import binding as B
from paper_2608_12932_b200 import workload as wl
from tests.gpu_util import bits, t_u16

pytestmark = pytest.mark.gpu


def bf16_bits(a):
    return bits(torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda().bfloat16())


@pytest.mark.parametrize("M", [1, 8, 16])
def test_a_used_workspace_gives_the_bits_of_a_fresh_one(M):
    I, K = 256, 256
    case = wl.make_layer(K, 2 * I, 11, 4)
    packed = B.w4a8_pack_weights(torch.from_numpy(case["qw"]).cuda(), t_u16(case["sw"], torch.float16), torch.from_numpy(case["z"]).cuda())
    rng = np.random.default_rng(5)
    used = B.new_workspace(16, 2 * I, K)

    def call(x_bits, ws, form):
        q = B.w4a8_quantize_act(t_u16(x_bits, torch.bfloat16))
        out = B.w4a8_gate_up_silu_quantize(*q, packed, 2 * I, ws, form=form)
        B.w4a8_check_status(ws)
        return out

    small = rng.standard_normal((M, K)) * 0.01
    small[M // 2] = 0.0                                        # a token whose h is zero throughout: no maximum is ever written
    small = bf16_bits(small)
    for form in (B.GATE_UP_EPILOGUE, B.GATE_UP_ONE_KERNEL, B.GATE_UP_EPILOGUE, B.GATE_UP_ONE_KERNEL):
        call(bf16_bits(rng.standard_normal((16, K)) * 100.0), used, form)
        for repeat in range(2):
            got, fresh = call(small, used, form), call(small, B.new_workspace(16, 2 * I, K), form)
            for a, b in zip(got, fresh):
                assert torch.equal(a.view(torch.uint8) if a.dtype != torch.int32 else a, b.view(torch.uint8) if b.dtype != torch.int32 else b)
            qa, sa, asum = onp.quantize_act(bits(got[0]), 128)
            assert np.array_equal(got[1].cpu().numpy(), qa) and np.array_equal(bits(got[2]), sa) and np.array_equal(got[3].cpu().numpy(), asum)
            assert bits(got[2])[M // 2] == 0


def layers(I, K):
    gu, down = wl.make_layer(K, 2 * I, 11, 4), wl.make_layer(I, K, 12, 4)
    return [B.w4a8_pack_weights(torch.from_numpy(c["qw"]).cuda(), t_u16(c["sw"], torch.float16), torch.from_numpy(c["z"]).cuda()) for c in (gu, down)]


def workspace(I, K):
    return max((B.new_workspace(16, *nk) for nk in ((2 * I, K), (K, I))), key=lambda w: w.numel())


def step(x, gu, down, I, K, ws, form, other):
    """One fused step and the down projection behind it; `other`: a call of another kernel family on the workspace between them."""
    q = B.w4a8_quantize_act(x)
    out = B.w4a8_gate_up_silu_quantize(*q, gu, 2 * I, ws, form=form)
    if other:
        B.w4a8_gemm(*q, gu, 2 * I, ws, path=other)
    return [*out, B.w4a8_gemm(*out[1:], down, K, ws)]


@pytest.mark.parametrize("form", [B.GATE_UP_EPILOGUE, B.GATE_UP_ONE_KERNEL])
def test_what_a_call_leaves_in_the_workspace(form):
    """As the public header says it: bytes 64 to 207 hold maxima and call numbers, all else of the zeroed part is zero again."""
    I, K = 6144, 1280
    gu, down = layers(I, K)
    ws = workspace(I, K)
    rng = np.random.default_rng(3)
    for M in (16, 5, 8):
        step(t_u16(bf16_bits(rng.standard_normal((M, K))), torch.bfloat16), gu, down, I, K, ws, form, None)
    B.w4a8_check_status(ws)
    left = ws[:4096 + 192 * 16384].cpu().numpy()
    words = left[64:208].view(np.uint64)
    assert (words[:16] >> np.uint64(16)).max() == 3 and (words[:16] & np.uint64(0xFFFF)).all() and words[16] == 3
    assert not left[:64].any() and not left[208:].any()


def same(got, want):
    return all(torch.equal(a.view(torch.uint8), b.view(torch.uint8)) for a, b in zip(got, want, strict=True))


# 1280 -> 2 x 6144: 384 strips of 32 channels in two stages each, more than there are CTAs, so that neighbours share strips
@pytest.mark.parametrize("M,I,K", [(1, 256, 256), (8, 256, 256), (16, 2432, 1024), (1, 6144, 1280), (8, 6144, 1280), (16, 6144, 1280)])
def test_steps_behind_one_another(M, I, K):
    """Nothing waits on the host between the calls, so a call's kernels start while the last call's still run: large and small
    values, both token counts, both forms and other kernel families in turn, then the same captured and replayed."""
    plan = B.w4a8_plan(M, 2 * I, K)
    if I == 6144 and M <= 8:
        assert plan["strip_rows"] == 32 and any(768 * c // plan["ctas"] % 2 for c in range(plan["ctas"]))
    gu, down = layers(I, K)
    rng = np.random.default_rng(M + I)
    bf = lambda m, scale: t_u16(bf16_bits(rng.standard_normal((m, K)) * scale), torch.bfloat16)
    seq = [(bf(16, 100.0), B.GATE_UP_EPILOGUE, None), (bf(M, 0.01), B.GATE_UP_EPILOGUE, None), (bf(M, 1.0), B.GATE_UP_ONE_KERNEL, None),
           (bf(M, 0.01), B.GATE_UP_EPILOGUE, B.PATH_SPLITK), (bf(16, 10.0), B.GATE_UP_ONE_KERNEL, B.PATH_TCGEN05),
           (bf(M, 0.1), B.GATE_UP_ONE_KERNEL, None), (bf(M, 0.01), B.GATE_UP_EPILOGUE, B.PATH_TCGEN05), (bf(M, 0.02), B.GATE_UP_EPILOGUE, None)]
    if M > 1:
        for x, _, _ in seq[1:]:
            x[x.shape[0] // 2] = 0                             # a token whose h is zero throughout leaves its old maximum in place
    want = []
    for x, form, other in seq:
        ws = workspace(I, K)
        want.append(step(x, gu, down, I, K, ws, form, other))
        B.w4a8_check_status(ws)
    assert all(bits(w[2]).any() for w in want)                 # scales of h that are not zero: maxima were written
    used = workspace(I, K)
    torch.cuda.synchronize()
    got = [step(x, gu, down, I, K, used, form, other) for _ in range(3) for x, form, other in seq]
    B.w4a8_check_status(used)
    assert all(same(g, want[i % len(seq)]) for i, g in enumerate(got))

    x = seq[1][0].clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = [step(x, gu, down, I, K, used, form, None) for form in (B.GATE_UP_EPILOGUE, B.GATE_UP_ONE_KERNEL, B.GATE_UP_EPILOGUE)]
    pick = [k for k in range(len(seq)) if seq[k][0].shape[0] == M]
    kept = []
    for k in pick * 2:
        x.copy_(seq[k][0])
        graph.replay()
        kept.append((k, [[t.clone() for t in o] for o in out]))
    B.w4a8_check_status(used)
    for k, outs in kept:
        assert all(same(o, want[k]) for o in outs), k

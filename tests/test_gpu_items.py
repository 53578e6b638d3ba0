"""The matrix queue's items where its rules change: column tiles of long experts, strips cut into pieces, items taken in
batches, the combine order's token limit; and host buffers that are not pinned."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2605_23764_b200 import MoeLayer, binding as B
from tests.gpu_util import assert_close_bf16, small_problem

pytestmark = pytest.mark.gpu


def _against_oracle(ids, w, x, W1, W2, dout, serial):
    T, d = x.shape
    E, F = W2.shape[0], W2.shape[2]
    layer = MoeLayer(T, d, E, ids.shape[1], 0, F, save_for_bwd=True, serial=serial)
    out = layer.ffn_fwd(x, ids, w, W1, W2)
    dx, dW1, dW2, dw = layer.ffn_bwd(dout, x, ids, w, W1, W2)
    torch.cuda.synchronize()
    assert layer.status() == (0, 0)
    assert_close_bf16(out, oracle.fwd(x, ids.cpu(), w.cpu(), W1, W2), "out")
    rdx, rdW1, rdW2, rdw = oracle.bwd(dout, x, ids.cpu(), w.cpu(), W1, W2)
    assert_close_bf16(dx, rdx, "dx")
    assert_close_bf16(dw, rdw, "d_topk_w")
    for e in range(E):   # expert by expert: a tile left out would hide in the whole tensors' norms
        if (ids == e).any():
            assert_close_bf16(dW1[e], rdW1[e], f"dW_gate_up[{e}]")
            assert_close_bf16(dW2[e], rdW2[e], f"dW_down[{e}]")
        else:
            assert torch.count_nonzero(dW1[e]).item() == 0 and torch.count_nonzero(dW2[e]).item() == 0
    layer.close()


@pytest.mark.parametrize("counts,d,F", [
    ([960, 961, 0, 40], 1320, 72),       # the last resident-strip expert and the first long one; fewer strips than pairs
    ([1025, 320, 321, 7], 520, 392),     # a long expert beside strips that stay resident and that do not
])
@pytest.mark.parametrize("serial", [False, True])
def test_weight_gradient_items(counts, d, F, serial):
    E, T = len(counts), sum(counts)
    g = torch.Generator().manual_seed(T)
    ids = torch.from_numpy(np.repeat(np.arange(E), counts).astype(np.int32))[torch.randperm(T, generator=g)].reshape(T, 1)
    w = torch.rand(T, 1, generator=g) + 0.25
    x, W1, W2, _, dout = small_problem(T, d, E, 1, 0, F, T)
    _against_oracle(ids.contiguous().cuda(), w.cuda(), x, W1, W2, dout, serial)


@pytest.mark.parametrize("d", [4096, 2048])   # 20 and 10 items of one k-block to a CTA pair: batches of four and of two
def test_short_items_in_batches(d):
    T, E, k, F = 640, 96, 3, 64
    x, W1, W2, logits, dout = small_problem(T, d, E, k, 0, F, d)
    layer = MoeLayer(T, d, E, k, 0, F)
    ids, w = layer.route(logits)
    torch.cuda.synchronize()
    layer.close()
    _against_oracle(ids, w, x, W1, W2, dout, False)


@pytest.mark.parametrize("T", [511, 512, 513])
def test_combine_with_and_without_an_order(T):
    d, E, k, S, F = 136, 12, 3, 1, 72
    x, W1, W2, logits, _ = small_problem(T, d, E, k, S, F, T)
    outs = []
    for serial in (False, True):
        layer = MoeLayer(T, d, E, k, S, F, serial=serial)
        ids, w = layer.route(logits)
        outs.append(layer.ffn_fwd(x, ids, w, W1, W2).clone())
        assert layer.status() == (0, 0)
        layer.close()
    assert torch.equal(*outs)   # the same sums in slot order


def test_host_buffers_that_are_not_pinned():
    T, d, E, k, S, F = 300, 136, 12, 3, 1, 72
    x, W1, W2, logits, dout = small_problem(T, d, E, k, S, F, 3)
    res = []
    for pin in (True, False):
        def host(t):
            return t.cpu().pin_memory() if pin else t.cpu()
        def empty(*shape, dtype):
            return torch.empty(*shape, dtype=dtype, pin_memory=pin)
        layer = MoeLayer(T, d, E, k, S, F, save_for_bwd=True)
        ids, w, dw = empty(T, k, dtype=torch.int32), empty(T, k, dtype=torch.float32), empty(T, k, dtype=torch.float32)
        out, dx = empty(T, d, dtype=torch.bfloat16), empty(T, d, dtype=torch.bfloat16)
        dW1, dW2 = torch.empty_like(W1), torch.empty_like(W2)
        B.moe_route_host(layer.ctx, host(logits), T, ids, w)
        torch.cuda.synchronize()
        B.moe_ffn_fwd_host(layer.ctx, host(x), ids, w, W1, W2, out, T)
        torch.cuda.synchronize()
        B.moe_ffn_bwd_host(layer.ctx, host(dout), W1, W2, dx, dW1, dW2, dw, T)
        torch.cuda.synchronize()
        assert layer.status() == (0, 0)
        res.append((ids, w, out, dx, dw, dW1, dW2))
        layer.close()
    assert all(torch.equal(a, b) for a, b in zip(*res))


@pytest.mark.parametrize("case", ["one_expert", "padded_batch", "merged"])
@pytest.mark.parametrize("serial", [False, True])
def test_ids_repeated_inside_a_token(case, serial):
    """An expert may have more rows than the call has tokens: every slot of a token is a row of its own."""
    d, E, F = 1032, 8, 392   # 17 and 7 k-blocks: more than the deepest ring has stages, and fewer
    if case == "one_expert":       # 32 tokens x 8 slots, all of them expert 0's
        T, k = 32, 8
        ids = torch.zeros(T, k, dtype=torch.int32)
    elif case == "padded_batch":   # half of a generation batch is padding with id 0 in every slot
        T, k = 64, 6
        ids = torch.stack([torch.randperm(E, generator=torch.Generator().manual_seed(t))[:k] for t in range(T)]).to(torch.int32)
        ids[T // 2:] = 0
    else:                          # 256 tokens: experts of 290 and 222 rows, the larger one's last two tiles merge
        T, k = 256, 2
        ids = torch.zeros(T, k, dtype=torch.int32)
        ids[145:, :] = 3
    w = torch.rand(T, k, generator=torch.Generator().manual_seed(T)) + 0.25
    x, W1, W2, _, dout = small_problem(T, d, E, k, 0, F, T)
    _against_oracle(ids.cuda(), w.cuda(), x, W1, W2, dout, serial)


def test_host_memory_is_used_in_place_only_within_one_registration():
    """Looked up only: no kernel touches the memory."""
    mb, rt = 1 << 20, torch.cuda.cudart()
    torch.zeros(1, device="cuda")
    pinned, pageable = torch.empty(mb, dtype=torch.uint8, pin_memory=True), torch.empty(9 * mb, dtype=torch.uint8)
    assert B.moe_debug_host_direct(pinned.data_ptr(), mb) and B.moe_debug_host_direct(pinned.data_ptr() + mb - 4, 4)
    assert not B.moe_debug_host_direct(pageable.data_ptr(), mb)
    first = (pageable.data_ptr() + mb - 1) // mb * mb
    second = first + 4 * mb
    assert not int(rt.cudaHostRegister(first, mb, 0)) and not int(rt.cudaHostRegister(second, mb, 0))
    try:
        assert B.moe_debug_host_direct(first, mb) and B.moe_debug_host_direct(second + 4, mb - 4)
        assert not B.moe_debug_host_direct(first, mb + 4)       # beyond the end
        assert not B.moe_debug_host_direct(first, 5 * mb)       # both ends registered, a gap between them
    finally:
        rt.cudaHostUnregister(first)
        rt.cudaHostUnregister(second)


def test_workspace_views_of_one_context_stay_apart():
    """Rows of 136 and 72 columns are padded in the workspace: each tensor's compact copy stays while others are asked for."""
    T, d, E, k, S, F = 70, 136, 5, 2, 1, 72
    x, W1, W2, logits, _ = small_problem(T, d, E, k, S, F, 12)
    layer = MoeLayer(T, d, E, k, S, F, save_for_bwd=True)
    ids, w = layer.route(logits)
    layer.ffn_fwd(x, ids, w, W1, W2)
    names = ("Xp", "Y", "A", "H")
    want = [layer.debug(n) for n in names]
    views = []
    for n in names:
        ptr, elems = ctypes.c_void_p(), ctypes.c_size_t()
        assert B.load_library().moe_debug_buffer(layer.ctx, B.MOE_BUF[n], ctypes.byref(ptr), ctypes.byref(elems)) == 0
        views.append(torch.as_tensor(B._DevView(ptr.value, elems.value, "<i2"), device="cuda"))
    rows = (layer.debug("prow_of")[:T * (k + S)].long(), )
    for n, v, t, cols in zip(names, views, want, (d, d, F, 2 * F)):
        assert torch.equal(v.view(-1, cols)[rows], t.view(torch.int16).view(-1, cols)[rows]), n
    layer.close()


@pytest.mark.parametrize("T", [1, 70, 300])
def test_event_counters_as_documented(T):
    """moe_debug_buffer's view of the event counters, which lie apart in the workspace: eight words, then {gathered, activated,
    done, 0} of each M-block -- after a forward, and again after a backward, at their thresholds."""
    d, E, k, S, F = 264, 5, 2, 1, 136
    x, W1, W2, logits, dout = small_problem(T, d, E, k, S, F, 12)
    layer = MoeLayer(T, d, E, k, S, F, save_for_bwd=True)
    ids, w = layer.route(logits)

    def expect(col_tiles_first, col_tiles_last):
        counts = layer.debug("counts").cpu().numpy()
        want = []
        for n in counts:
            n32 = (int(n) + 31) // 32 * 32
            want += [[min(128, n32 - r) // 4, 2 * col_tiles_first, 2 * col_tiles_last, 0] for r in range(0, int(n), 128)]
        got = layer.debug("event_counters").cpu()
        assert got[1] == 0   # no trace
        assert got[8:8 + 4 * len(want)].reshape(-1, 4).tolist() == want
        assert torch.count_nonzero(got[8 + 4 * len(want):]).item() == 0

    layer.ffn_fwd(x, ids, w, W1, W2)
    torch.cuda.synchronize()
    expect((F + 127) // 128, (d + 255) // 256)
    layer.ffn_bwd(dout, x, ids, w, W1, W2)
    torch.cuda.synchronize()
    expect((F + 255) // 256, (d + 255) // 256)
    layer.close()

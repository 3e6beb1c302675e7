"""The native per-call module (csrc/py_calls.cpp): it declines (None) whatever is not the plain valid case, so that the
Python binding raises its own error, and gives the Python binding's results otherwise.  An int `scale` is one of the
arguments it declines: the same value as int and as float takes the two routes."""
import ctypes
import os
import subprocess
import sys
import threading

import pytest
import torch

import paper_2605_05838_b200 as mdn


def args(B, T, H, dk, dv, dtype, device, seed=0):
    g = torch.Generator().manual_seed(seed)
    q, k = (torch.nn.functional.normalize(torch.randn((B, T, H, dk), generator=g), dim=-1).to(dtype) for _ in range(2))
    v = torch.randn((B, T, H, dv), generator=g).to(dtype)
    beta = torch.rand((B, T, H), generator=g) * 0.05
    la, lm = (-0.1 * torch.rand((B, T, H), generator=g) for _ in range(2))
    eta = 1.0 + 0.1 * torch.randn((B, T, H), generator=g)
    return [t.to(device) for t in (q, k, v, beta, la, lm, eta)]


def test_cpu_tensors_are_declined_and_the_binding_raises():
    from paper_2605_05838_b200 import build
    build.build()
    from paper_2605_05838_b200.binding import _load_native
    a = args(1, 1, 2, 64, 64, torch.float32, "cpu")
    S = torch.zeros((1, 2, 64, 64))
    nat = _load_native()
    assert nat.decode_step(*a, S, S, None, None, None, 0) is None
    assert nat.chunk_fwd(*a, None, None, None, None, None, 0, True, None, None, 0, 0, False) is None
    assert nat.chunk_bwd(*a, a[2], None, None, None, None, None, None, None, 0, None, None) is None
    ops = mdn.MdnLayerOps()
    assert nat.fill_layer_ops(ctypes.addressof(ops), a[0], a[2], None, None, None, "fused") is None
    for call in (lambda: mdn.decode_step(*a, S, S), lambda: mdn.chunk_fwd(*a), lambda: mdn.chunk_bwd(*a, a[2])):
        with pytest.raises(ValueError):
            call()
    with pytest.raises(KeyError):
        mdn.make_layer_ops(a[0], a[2], placement="nosuch")


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,dk,dv,T", [(torch.float32, 64, 128, 1), (torch.float32, 64, 64, 65), (torch.bfloat16, 128, 128, 70)])
def test_both_routes_give_the_same_bits(dtype, dk, dv, T):
    a = args(2, T, 3, dk, dv, dtype, "cuda")
    g = torch.Generator().manual_seed(5)
    S, M = (torch.randn((2, 3, dk, dv), generator=g).cuda() * 0.1 for _ in range(2))
    for kw in (dict(), dict(initial_S=S, initial_M=M, o_dtype=torch.float32), dict(output_final_state=False)):
        for x, y in zip(mdn.chunk_fwd(*a, scale=1, **kw), mdn.chunk_fwd(*a, scale=1.0, **kw)):
            assert (x is None and y is None) or torch.equal(x, y)
    if T == 1:
        S2, M2 = S.clone(), M.clone()
        o1, o2 = mdn.decode_step(*a, S, M, scale=1), mdn.decode_step(*a, S2, M2, scale=1.0)
        assert torch.equal(o1, o2) and torch.equal(S, S2) and torch.equal(M, M2)
    d_o = a[2].clone()
    g1, g2 = mdn.chunk_bwd(*a, d_o, scale=1), mdn.chunk_bwd(*a, d_o, scale=1.0)
    assert g1.keys() == g2.keys() and torch.equal(g1["dv"], g2["dv"]) and torch.equal(g1["d_initial_S"], g2["d_initial_S"])
    with pytest.raises(mdn.MdnError):
        mdn.chunk_fwd(*a, scale=1.0, segments=2)


@pytest.mark.gpu
def test_kernels_run_after_a_device_reset():
    """The kernels' shared-memory limits are gone with the old context and set anew."""
    child = os.path.join(os.path.dirname(os.path.abspath(__file__)), "probe", "reset_child.py")
    r = subprocess.run([sys.executable, child], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "[0, 0, 0, 0]", r.stdout + r.stderr


@pytest.mark.gpu
def test_threads_that_launch_one_kernel_with_different_sizes():
    """The fp32 kernels take more shared memory for bf16 input and wider values: threads that use both at the same time."""
    errors = []

    def work(dtype, dv, stream):
        try:
            with torch.cuda.stream(stream):
                a = args(1, 70, 2, 128, dv, dtype, "cuda")
                want = mdn.chunk_fwd(*a, path="simt")[0]
                for _ in range(200):
                    assert torch.equal(mdn.chunk_fwd(*a, path="simt")[0], want)
                    mdn.chunk_bwd(*a, a[2])
                stream.synchronize()
        except Exception as e:   # handed to the test's thread
            errors.append(e)
    threads = [threading.Thread(target=work, args=(dt, dv, torch.cuda.Stream()))
               for dt in (torch.float32, torch.bfloat16) for dv in (64, 128)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def misaligned(t):
    """The same values in a contiguous tensor that starts two bytes behind a 16-byte boundary."""
    buf = torch.empty(t.numel() + 8, dtype=t.dtype, device=t.device)
    m = buf[1:1 + t.numel()].view(t.shape)
    return m.copy_(t)


def attention_args(T=100):
    return [t.requires_grad_() for t in args(1, T, 2, 128, 128, torch.bfloat16, "cuda")]


@pytest.mark.gpu
def test_a_refused_call_of_the_differentiable_forward_is_an_MdnError():
    """In the forward (q) and, through the autograd engine's thread, in the backward (d_o)."""
    a = attention_args()
    with pytest.raises(mdn.MdnError) as e:
        mdn.chunk_attention(misaligned(a[0].detach()), *a[1:])
    assert e.value.status == 1
    o, _, _ = mdn.chunk_attention(*a)
    with pytest.raises(mdn.MdnError) as e:
        torch.autograd.grad(o, a, misaligned(torch.ones_like(o)))
    assert e.value.status == 1


@pytest.mark.gpu
def test_exceptions_of_saved_tensor_hooks_pass_through():
    class Mine(Exception):
        pass

    def fail(_):
        raise Mine("hook")
    a = attention_args()
    with pytest.raises(Mine), torch.autograd.graph.saved_tensors_hooks(fail, lambda x: x):
        mdn.chunk_attention(*a)
    with torch.autograd.graph.saved_tensors_hooks(lambda x: x, fail):
        o, _, _ = mdn.chunk_attention(*a)
    with pytest.raises(Mine):
        o.float().sum().backward()


def grads_of(run, a):
    o, S, _ = run(*a)
    return torch.autograd.grad(o.float().square().sum() + S.square().sum(), a)


def same_gradients(x, y):   # (gate gradients: sums by atomics, last bits may differ)
    return all(torch.equal(u, w) if u.dtype == torch.bfloat16 else (u - w).abs().max() <= 1e-4 * w.abs().max() for u, w in zip(x, y))


@pytest.mark.gpu
def test_activation_checkpointing():
    """The recomputation ends with an exception out of the last saved tensor's hook, which the checkpoint catches."""
    from torch.utils.checkpoint import checkpoint
    a = attention_args()
    want = grads_of(mdn.chunk_attention, a)
    assert same_gradients(grads_of(lambda *x: checkpoint(mdn.chunk_attention, *x, use_reentrant=False), a), want)


@pytest.mark.gpu
def test_saved_tensors_that_come_back_elsewhere():
    """Hooks that keep the saved tensors on the host (or copy them): the kept states need their 1024-byte boundary again.  What comes
    back in other strides or another type is refused."""
    a = attention_args()
    want = grads_of(mdn.chunk_attention, a)
    with torch.autograd.graph.save_on_cpu(pin_memory=True):
        assert same_gradients(grads_of(mdn.chunk_attention, a), want)

    def shifted(t):   # every byte buffer 256 bytes behind a 1024-byte boundary
        if t.dtype != torch.uint8:
            return t.clone()
        buf = torch.empty(t.numel() + 2048, dtype=t.dtype, device=t.device)
        at = -buf.data_ptr() % 1024 + 256
        return buf[at:at + t.numel()].copy_(t)
    with torch.autograd.graph.saved_tensors_hooks(shifted, lambda x: x):
        assert same_gradients(grads_of(mdn.chunk_attention, a), want)
    for bad in (lambda t: t.transpose(1, 2).contiguous().transpose(1, 2), lambda t: t.float()):
        change = lambda t: bad(t) if t.dim() == 4 and t.dtype == torch.bfloat16 else t
        with torch.autograd.graph.saved_tensors_hooks(change, lambda x: x):
            o, _, _ = mdn.chunk_attention(*a)
        with pytest.raises(ValueError):
            o.float().sum().backward()

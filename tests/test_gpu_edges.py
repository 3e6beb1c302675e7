"""Sizes at which the kernels' splits change: rows per tile of the exact backward (up to 32 tokens / more), value columns
per CTA of the fp32 chains (8 while that makes at most 148 CTAs, else 16), the uneven segments of the parallel
inter-chunk scan, and the two routes of the differentiable forward."""
import ctypes

import numpy as np
import pytest

import mdn_workloads as wl
from helpers import rel_err, run_gpu, run_oracle, to_torch
from test_gpu_bwd import check, run_both, upstream

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mdn():
    import paper_2605_05838_b200 as m
    m.lib()
    return m


@pytest.mark.parametrize("B,H,dk,dv,T,dtype", [
    (1, 1, 64, 64, 31, "f32"), (1, 1, 128, 64, 32, "f32"), (1, 2, 64, 128, 33, "bf16"),
    (1, 9, 128, 128, 129, "f32"),       # 9 heads x 16 blocks of 8 columns = 144 CTAs
    (1, 10, 128, 128, 65, "f32"),       # 160: 16 columns per CTA
    (2, 10, 64, 64, 97, "f32")])
def test_exact_backward_tiles(mdn, B, H, dk, dv, T, dtype):
    """fp32 arithmetic throughout: the bound of the exact backward (1e-4 of RMS)."""
    w = wl.Workload("edge_bwd", B=B, T=T, H=H, dk=dk, dv=dv, dtype=dtype, init_state_std=0.2, seed=T)
    inp = wl.make_inputs(w)
    got, ref = run_both(mdn, inp, *upstream(w, inp, T))
    check(got, ref, "T=%d dk=%d dv=%d H=%d" % (T, dk, dv, H))


@pytest.mark.parametrize("H,dv,T", [(9, 128, 130), (10, 128, 70), (18, 64, 64), (19, 64, 65)])
def test_fp32_chain_columns_per_cta(mdn, H, dv, T):
    """On either side of the 148-CTA switch (144 / 160, 144 / 152) the split meets the fp32 bound (1e-4), and gives the bits of one head
    alone, which takes the narrow one (the sums are split alike)."""
    w = wl.Workload("edge_simt", B=1, T=T, H=H, dk=64, dv=dv, dtype="f32", init_state_std=0.2, seed=H)
    inp = wl.make_inputs(w)
    o, S, M = run_gpu(mdn, inp, path="simt")
    o_ref, S_ref, M_ref = run_oracle(inp)
    assert max(rel_err(o, o_ref), rel_err(S, S_ref), rel_err(M, M_ref)) <= 1e-4
    t = to_torch(inp)
    part = lambda x: x[:1, :, :1].contiguous()
    g = [part(t[n]) for n in ("q", "k", "v", "beta", "log_alpha", "log_mu", "eta")]
    o1, S1, M1 = mdn.chunk_fwd(*g, initial_S=t["initial_S"][:1, :1].contiguous(), initial_M=t["initial_M"][:1, :1].contiguous(),
                               scale=inp["scale"], path="simt")
    assert np.array_equal(o1.cpu().numpy()[0, :, 0], np.asarray(o)[0, :, 0])
    assert np.array_equal(S1.cpu().numpy()[0, 0], np.asarray(S)[0, 0]) and np.array_equal(M1.cpu().numpy()[0, 0], np.asarray(M)[0, 0])


@pytest.mark.parametrize("B,H,T", [(1, 1, 64 * 51 + 17), (2, 2, 64 * 61), (1, 8, 64 * 90 + 1)])
def test_automatic_segments(mdn, B, H, T):
    """Few long chains are split by rule into unequal segments: same recurrence within the bf16 path's bound, and the first
    segment's tokens come from the same run as the serial chain's."""
    import torch
    w = wl.Workload("edge_seg", B=B, T=T, H=H, dk=128, dv=128, dtype="bf16", init_state_std=0.3, seed=T)
    lay = mdn.workspace_layout(mdn.MdnParams(B, T, H, 128, 128, 64, 0, 1, 0, 0, 1.0, 0))
    assert lay.segments > 1
    inp = wl.make_inputs(w)
    o_ref, S_ref, M_ref = run_oracle(inp)
    o, S, M = run_gpu(mdn, inp, path="tensor", o_dtype=torch.float32)
    assert max(rel_err(o, o_ref), rel_err(S, S_ref), rel_err(M, M_ref)) <= 2e-2
    o1, _, _ = run_gpu(mdn, inp, path="tensor", o_dtype=torch.float32, segments=1)
    assert np.array_equal(np.asarray(o)[:, :64], np.asarray(o1)[:, :64])


@pytest.mark.parametrize("segments,H,lens", [(0, 1, [64 * 200 + 5, 64 * 33, 100, 64 * 140 + 63, 1]), (3, 2, [64 * 3, 64 * 2 + 1, 1, 64 * 9 + 7]),
                                             (0, 2, [63, 64 * 150])])
def test_segments_of_packed_sequences(mdn, segments, H, lens):
    """Packed sequences are split in proportion to their lengths; those too short for it stay whole (empty segments behind)."""
    import torch
    w = wl.Workload("edge_pseg", B=1, T=sum(lens), H=H, dk=128, dv=128, dtype="bf16", varlen=True, init_state_std=0.3, seed=len(lens))
    assert mdn.workspace_layout(mdn.MdnParams(1, w.T, H, 128, 128, 64, len(lens), 1, 0, 0, 1.0, segments)).segments > 1
    inp = wl.make_inputs(w, lengths=np.array(lens))
    o_ref, S_ref, M_ref = run_oracle(inp)
    o, S, M = run_gpu(mdn, inp, path="tensor", o_dtype=torch.float32, segments=segments)
    assert max(rel_err(o, o_ref), rel_err(S, S_ref), rel_err(M, M_ref)) <= 2e-2


@pytest.mark.parametrize("B,H,T,lens", [(1, 1, 64 * 45 + 17, None), (2, 2, 64 * 40, None), (1, 1, 0, [64 * 110 + 3, 64 * 40, 70])])
def test_training_with_segments(mdn, B, H, T, lens):
    """Few long chains: both chains of a training step are split as the forward is.  Against the exact fp32 backward (1e-4 of the
    oracle): the tensor-core backward's bounds, 2e-2 of RMS per element (dv 3e-2: largest of 1e5 .. 1e6 values rounded to bf16 on the
    way, the serial chain's own is 2.1e-2 here and up to 2.8e-2 elsewhere) and 5e-3 in RMS."""
    import torch
    w = wl.Workload("edge_tseg", B=B, T=T or sum(lens), H=H, dk=128, dv=128, dtype="bf16", varlen=lens is not None, init_state_std=0.1, seed=B + 7)
    assert mdn.workspace_layout(mdn.MdnParams(B, w.T, H, 128, 128, 64, len(lens) if lens else 0, 1, 1, 0, 1.0, 0)).segments > 1
    t = to_torch(wl.make_inputs(w, lengths=np.array(lens)) if lens else wl.make_inputs(w))
    d_o = torch.randn(t["v"].shape, generator=torch.Generator().manual_seed(4)).to(torch.bfloat16).cuda()
    args = (t["q"], t["k"], t["v"], t["beta"], t["log_alpha"], t["log_mu"], t["eta"])
    kw = dict(initial_S=t["initial_S"], initial_M=t["initial_M"], cu_seqlens=t["cu_seqlens"], scale=0.1)
    ref = mdn.chunk_bwd(*args, d_o, method="stepwise", **kw)
    _, _, _, states, ws = mdn.chunk_fwd(*args, path="tensor", keep_chunk_states=True, **kw)
    for saved in (None, (ws, states)):
        got = mdn.chunk_bwd(*args, d_o, method="chunked", saved=saved, **kw)
        for name, y in ref.items():
            x, y = got[name].double().cpu().numpy(), y.double().cpu().numpy()
            assert rel_err(x, y) <= (3e-2 if name == "dv" else 2e-2), name
            assert np.sqrt(np.mean((x - y) ** 2)) <= 5e-3 * np.sqrt(np.mean(y ** 2)), name


@pytest.mark.parametrize("packed,state,eta", [(False, True, True), (True, True, False), (False, False, False)])
def test_both_autograd_nodes_give_the_same_bits(mdn, packed, state, eta):
    """The C++ node and the Python one run the same kernels (gate gradients: sums by atomics, last bits may differ)."""
    import torch
    from paper_2605_05838_b200.binding import _ChunkAttention
    w = wl.Workload("edge_ag", B=1 if packed else 2, T=200, H=2, dk=128, dv=128, dtype="bf16", seed=7, varlen=packed, len_lo=20,
                    len_hi=90, init_state_std=0.2 if state else 0.0)
    t = to_torch(wl.make_inputs(w))
    names = ["q", "k", "v", "beta", "log_alpha", "log_mu"] + (["eta"] if eta else []) + (["initial_S", "initial_M"] if state else [])
    res = []
    for native in (True, False):
        x = {n: t[n].clone().requires_grad_(True) for n in names}
        kw = dict(initial_S=x.get("initial_S"), initial_M=x.get("initial_M"), cu_seqlens=t["cu_seqlens"])
        a = (x["q"], x["k"], x["v"], x["beta"], x["log_alpha"], x["log_mu"], x.get("eta"))
        if native:
            o, S, M = mdn.chunk_attention(*a, scale=0.1, **kw)
        else:
            o, S, M = _ChunkAttention.apply(*a, kw["initial_S"], kw["initial_M"], kw["cu_seqlens"], 0.1)
        (o.float().square().sum() + S.square().sum()).backward()
        res.append((o.detach(), S.detach(), M.detach()) + tuple(x[n].grad for n in names))
    for n, x, y in zip(["o", "S", "M"] + names, *res):
        if n in ("beta", "log_alpha", "log_mu", "eta"):
            assert (x - y).abs().max() <= 1e-4 * y.abs().max(), n
        else:
            assert torch.equal(x, y), n


@pytest.mark.parametrize("T,H,dtype", [(64, 1, "float32"), (1, 4, "float32"), (3000, 8, "float32"), (1, 64, "bfloat16")])
def test_output_gate_made_by_the_call_before(mdn, T, H, dtype):
    """The output step's gate is what the call just before wrote on the same stream (its last kernel lets the next ones in before it
    stores): the same bits as with a synchronisation between the two.  T = 1: also through decode_step."""
    import torch
    dt = getattr(torch, dtype)
    g = torch.Generator(device="cuda").manual_seed(T)
    r = lambda *s: torch.randn(s, device="cuda", generator=g)
    q, k, v = (x.to(dt) for x in (0.1 * r(2, T, H, 64), 0.1 * r(2, T, H, 64), r(2, T, H, 64)))
    gates = (0.1 * r(2, T, H).abs(), -r(2, T, H).abs(), -0.1 * r(2, T, H).abs(), 1 + 0.1 * r(2, T, H))
    step = lambda gate: mdn.make_layer_ops(q, v, out_norm_gate=dict(g=gate, eps=1e-5))
    S = r(2, H, 64, 64)
    calls = [lambda gate: mdn.chunk_fwd(q, k, v, *gates, layer_ops=step(gate))[0]]
    if T == 1:
        calls.append(lambda gate: mdn.decode_step(q, k, v, *gates, S.clone(), S.clone(), layer_ops=step(gate)))
    for call in calls:
        first = call(v)
        torch.cuda.synchronize()
        want = call(first)
        torch.cuda.synchronize()
        for _ in range(50):
            assert torch.equal(call(call(v)), want)


def test_workspace_enough_for_the_serial_chain(mdn):
    """A workspace kept for the largest call also serves the shorter ones that the scan would split (and need more for): the result of
    segments = 1, for every call that takes a workspace."""
    import torch
    byref = ctypes.byref
    L = mdn.lib()
    for lens, B, T, H in ((None, 1, 3000, 2), ([7000, 1900, 100], 1, 9000, 1)):
        w = wl.Workload("edge_ws", B=B, T=T, H=H, dk=128, dv=128, dtype="bf16", varlen=lens is not None, init_state_std=0.1, seed=3)
        inp = wl.make_inputs(w, lengths=np.array(lens)) if lens else wl.make_inputs(w)
        t = to_torch(inp)
        a = [t[n] for n in ("q", "k", "v", "beta", "log_alpha", "log_mu", "eta")]
        kw = dict(initial_S=t["initial_S"], initial_M=t["initial_M"], cu_seqlens=t["cu_seqlens"], scale=0.1)
        N = len(lens) if lens else 0
        p, p1 = (mdn.make_params(a[0], a[2], num_seqs=N, scale=0.1, segments=s) for s in (0, 1))
        assert mdn.workspace_layout(p).segments > 1
        buf = lambda n: torch.empty(int(n) + 1024, dtype=torch.uint8, device="cuda")
        cut = lambda b, n: b[-b.data_ptr() % 1024:][:int(n)]
        space = lambda n: cut(buf(n), n)
        same = lambda x, y: all(torch.equal(u, v) for u, v in zip(x, y))
        # the forward, alone and with the layer operations as passes of their own
        ops = mdn.make_layer_ops(a[0], a[2], qk_norm=dict(eps=1e-6), out_norm_gate=dict(g=a[2], eps=1e-5), placement="separate")
        for lo in (None, ops):
            one = mdn.chunk_fwd(*a, segments=1, layer_ops=lo, **kw)
            n = mdn.workspace_bytes(p1) if lo is None else L.mdn_chunk_fwd_fused_workspace_bytes(byref(p1), byref(lo))
            n0 = mdn.workspace_bytes(p) if lo is None else L.mdn_chunk_fwd_fused_workspace_bytes(byref(p), byref(lo))
            assert n < n0
            assert same(mdn.chunk_fwd(*a, workspace=space(n), layer_ops=lo, **kw), one)
            with pytest.raises(mdn.MdnError):
                mdn.chunk_fwd(*a, workspace=space(n - 256), layer_ops=lo, **kw)
            with pytest.raises(mdn.MdnError):
                mdn.chunk_fwd(*a, workspace=space(n), segments=4, layer_ops=lo, **kw)
        # host buffers
        h = {k: (v.cpu().pin_memory() if v is not None else None) for k, v in t.items()}
        ha = [h[n] for n in ("q", "k", "v", "beta", "log_alpha", "log_mu", "eta")]
        hkw = dict(initial_S=h["initial_S"], initial_M=h["initial_M"], cu_seqlens=h["cu_seqlens"], scale=0.1)
        got = mdn.chunk_fwd_host(*ha, arena=space(mdn.host_arena_bytes(p1)), **hkw)
        assert same([x.cuda() for x in got], mdn.chunk_fwd(*a, segments=1, **kw))
        # training: the backward with and without kept states
        d_o = torch.randn(a[2].shape, generator=torch.Generator().manual_seed(2)).to(torch.bfloat16).cuda()
        st = mdn.chunk_fwd(*a, path="tensor", keep_chunk_states=True, workspace=space(mdn.workspace_bytes(p1)), **kw)
        want = mdn.chunk_bwd(*a, d_o, method="stepwise", **kw)
        pb, pb1 = (mdn.make_params(a[0], a[2], num_seqs=N, scale=0.1, path="tensor", segments=s) for s in (0, 1))
        for saved, size in ((None, L.mdn_chunk_bwd_chunked_workspace_bytes), ((st[4], st[3]), L.mdn_chunk_bwd_saved_workspace_bytes)):
            assert size(byref(pb1)) < size(byref(pb))
            got = mdn.chunk_bwd(*a, d_o, method="chunked", saved=saved, workspace=space(size(byref(pb1))), **kw)
            for n in want:   # (5e-3 in RMS: the tensor-core backward's bound)
                x, y = got[n].double(), want[n].double()
                assert (x - y).norm() <= 5e-3 * y.norm(), n
            with pytest.raises(mdn.MdnError):
                mdn.chunk_bwd(*a, d_o, method="chunked", saved=saved, workspace=space(size(byref(pb1)) - 1024), **kw)


@pytest.mark.parametrize("lens", [[0, 0, 5, 0], [1, 0, 0, 0, 0], [0, 70, 0]])
def test_forced_segments_with_fewer_tokens_than_sequences(mdn, lens):
    """Such sequences stay whole: the serial chain's bits, and an empty one hands its start state on."""
    import torch
    N, H, T = len(lens), 2, sum(lens)
    g = torch.Generator(device="cuda").manual_seed(N)
    r = lambda *s: torch.randn(s, device="cuda", generator=g)
    a = [(0.1 * r(1, T, H, 128)).bfloat16(), (0.1 * r(1, T, H, 128)).bfloat16(), r(1, T, H, 128).bfloat16(),
         0.1 * r(1, T, H).abs(), -r(1, T, H).abs(), -0.1 * r(1, T, H).abs(), 1 + 0.1 * r(1, T, H)]
    S0, M0 = r(N, H, 128, 128), r(N, H, 128, 128)
    cu = torch.tensor(np.concatenate([[0], np.cumsum(lens)]), dtype=torch.int32, device="cuda")
    one, three = (mdn.chunk_fwd(*a, initial_S=S0, initial_M=M0, cu_seqlens=cu, path="tensor", segments=s) for s in (1, 3))
    assert torch.equal(one[0], three[0])
    for x, y, z in zip(one[1:], three[1:], (S0, M0)):
        for n in range(N):
            assert torch.equal(x[n], y[n]) and (lens[n] > 0 or torch.equal(y[n], z[n])), n


def training_tensors(T, H):
    import torch
    g = torch.Generator(device="cuda").manual_seed(T)
    r = lambda *s: torch.randn(s, device="cuda", generator=g)
    n = lambda x: (x / x.norm(dim=-1, keepdim=True)).bfloat16()
    return [n(r(1, T, H, 128)), n(r(1, T, H, 128)), r(1, T, H, 128).bfloat16(), 0.05 * r(1, T, H).abs(), -0.1 * r(1, T, H).abs(),
            -0.1 * r(1, T, H).abs(), 1 + 0.1 * r(1, T, H)]


def test_training_keeps_no_scan_scratch(mdn):
    """Between forward and backward a call that the scan splits holds what the serial chain holds: outputs, states, and the workspace
    without the segments' states."""
    import torch
    a = [t.requires_grad_() for t in training_tensors(3000, 2)]
    p, p1 = (mdn.make_params(a[0], a[2], path="tensor", segments=s) for s in (0, 1))
    scan = mdn.workspace_bytes(p) - mdn.workspace_bytes(p1)
    assert scan > 4 << 20
    torch.cuda.synchronize()
    before = torch.cuda.memory_allocated()
    o, S, M = mdn.chunk_attention(*a)
    held = torch.cuda.memory_allocated() - before
    kept = int(mdn.lib().mdn_chunk_states_bytes(ctypes.byref(p))) + mdn.workspace_bytes(p1) + sum(x.numel() * x.element_size() for x in (o, S, M))
    assert kept <= held <= kept + (2 << 20)   # (the allocator's rounding)
    o.float().sum().backward()
    ref = mdn.chunk_bwd(*(t.detach() for t in a), torch.ones_like(o), method="stepwise")
    for x, n in zip(a, ("dq", "dk", "dv", "dbeta", "dlog_alpha", "dlog_mu", "deta")):
        assert (x.grad.float() - ref[n]).norm() <= 5e-3 * ref[n].norm(), n   # 5e-3 in RMS: the tensor-core backward's bound


@pytest.mark.parametrize("dk,dv,dtype", [(64, 64, "f32"), (128, 128, "bf16"), (128, 64, "f32"), (64, 128, "bf16")])
@pytest.mark.parametrize("B,T,H", [(1, 1, 1), (2, 8, 3), (1, 9, 2), (3, 18, 5), (1, 19, 2), (1, 25, 1), (5, 36, 15), (2, 41, 35), (2, 56, 50),
                                   (1, 57, 100), (200, 5, 1)])
def test_exact_backward_of_short_sequences(mdn, B, T, H, dk, dv, dtype):
    """The lengths around which the exact backward goes token by token (sums of 4, blocks of 8 tokens, up to 18 .. 56 tokens by the number
    of CTAs and dk, more chains than CTAs): the fp32 bound, 1e-4 of RMS; all but the gates' gradients bit-reproducible."""
    import torch
    w = wl.Workload("edge_short", B=B, T=T, H=H, dk=dk, dv=dv, dtype=dtype, init_state_std=0.2, seed=T)
    inp = wl.make_inputs(w)
    got, ref = run_both(mdn, inp, *upstream(w, inp, T))
    check(got, ref, "short B=%d T=%d H=%d" % (B, T, H))
    t = to_torch(inp)
    a = [t[n] for n in ("q", "k", "v", "beta", "log_alpha", "log_mu", "eta")]
    x, y = (mdn.chunk_bwd(*a, t["v"], scale=0.1) for _ in range(2))
    assert all(torch.equal(x[n], y[n]) for n in ("dq", "dk", "dv", "d_initial_S", "d_initial_M"))


@pytest.mark.parametrize("lens", [[3, 9, 1], [2, 0, 5, 1], [100, 28, 29, 56, 57, 64, 0, 1] + [7] * 92, [2] * 300, [150, 70, 20]])
@pytest.mark.parametrize("dv", [64, 128])
def test_exact_backward_of_packed_short_sequences(mdn, lens, dv):
    """Packed input: every sequence by its own length, some by chunks and some token by token; the same as one by one, and in a workspace
    without room for the second kind (all by chunks) the same to rounding."""
    import torch
    N, H, T, dk = len(lens), 2, sum(lens), 128
    g = torch.Generator(device="cuda").manual_seed(N)
    r = lambda *s: torch.randn(s, device="cuda", generator=g)
    n = lambda x: x / x.norm(dim=-1, keepdim=True)
    a = [n(r(1, T, H, dk)), n(r(1, T, H, dk)), r(1, T, H, dv), 0.05 * r(1, T, H).abs(), -0.1 * r(1, T, H).abs(), -0.1 * r(1, T, H).abs(),
         1 + 0.1 * r(1, T, H)]
    d_o = r(1, T, H, dv)
    st = {k: 0.2 * r(N, H, dk, dv) for k in ("initial_S", "initial_M", "d_final_S", "d_final_M")}
    cu = torch.tensor(np.concatenate([[0], np.cumsum(lens)]), dtype=torch.int32, device="cuda")
    got = mdn.chunk_bwd(*a, d_o, cu_seqlens=cu, **st)

    def close(x, y, what):   # fp32 sums in another order
        assert float((x - y).norm()) <= 2e-5 * float(y.norm()), what
    for i in sorted(set(range(0, N, max(1, N // 8))) | set(range(min(N, 8)))):
        if lens[i] == 0:
            assert torch.equal(got["d_initial_S"][i], st["d_final_S"][i])
            continue
        t0, t1 = int(cu[i]), int(cu[i + 1])
        one = mdn.chunk_bwd(*[x[:, t0:t1].contiguous() for x in a], d_o[:, t0:t1].contiguous(), **{k: x[i:i + 1].contiguous() for k, x in st.items()})
        for k, x in one.items():
            close(got[k][i:i + 1] if k.startswith("d_init") else got[k][:, t0:t1], x, (k, i, lens[i]))
    if N == 100:   # both kinds (all short: the chunk form needs more)
        need = int(mdn.lib().mdn_chunk_bwd_workspace_bytes(ctypes.byref(mdn.make_params(a[0], a[2], num_seqs=N))))
        fewer = mdn.chunk_bwd(*a, d_o, cu_seqlens=cu, workspace=torch.empty(need - 256, dtype=torch.uint8, device="cuda"), **st)
        for k in got:
            close(fewer[k], got[k], k)

"""GPU parity of kernel variants at the sizes where their dispatch or tiling changes, against the oracle."""
import numpy as np
import pytest
import torch

import oracle as vo
import paper_2504_18547_b200 as vt
import synth_inputs as si
from oracle import pipeline as vp
from gpu_util import GELU_TOL_REL, dev, from_codes, padding_is_zero, rand_codes, to_codes

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _device_status_clean():
    yield
    assert vt.vitint_device_status() == 0


def byte_codes(q, bits, signed):
    return to_codes(q, bits, signed) if bits == 8 else vt.vitint_widen(to_codes(q, bits, signed))


# ---- byte-stored operands, whole column blocks: single rows, row remainders of a 16-row unit and of a tile, one and
# ---- several column blocks, a last tile narrower than the others, K remainders of a block and of an MMA step
@pytest.mark.parametrize("M,K,N", [(1, 64, 64), (17, 48, 128), (127, 144, 320), (129, 768, 192), (145, 1000, 576), (1576, 320, 1088),
                                   (2600, 768, 2304)])
@pytest.mark.parametrize("bits", [2, 3, 4, 8])
def test_linear_direct_epilogues(M, K, N, bits):
    qx, qw = rand_codes(101 + M, (M, K), bits, True), rand_codes(102 + N, (N, K), bits, True)
    x, w = byte_codes(qx, bits, True), byte_codes(qw, bits, True)
    acc = vo.matmul_i32(qx, qw)
    spread = max(float(np.abs(acc).mean()), 1.0)
    s_w = ((np.abs(si.normal(103, (N,), 0.0, 0.2)) + 0.5) / spread).astype(np.float32)
    bias, res = si.normal(104, (N,), 0.0, 0.3), si.normal(105, (M, N))
    alpha, beta = s_w * np.float32(2 ** (bits - 1)), bias
    for cont, pitch in ((8, None), (0, None), (8, N + 48)):
        out = vt.Codes.empty(M, N, bits, True, container=cont, pitch=pitch)
        out.data.fill_(0xA5)
        vt.vitint_linear(x, 1.0, w, None, None, vt.Epilogue(mode=vt.EPI_REQUANT, alpha=dev(alpha), beta=dev(beta), out_bits=bits,
                                                            out_signed=True, out_container=cont), out=out)
        assert np.array_equal(from_codes(out), vo.epilogue_requant(acc, alpha, beta, bits, True)) and padding_is_zero(out)
    for r in (None, res):
        y = vt.vitint_linear(x, 0.75, w, dev(s_w), dev(bias), vt.Epilogue(mode=vt.EPI_DEQUANT_F32, residual=dev(r)))
        want = vo.epilogue_dequant(acc, np.float32(0.75), s_w, bias, r)
        assert np.array_equal(y.cpu().numpy().view(np.uint32), want.view(np.uint32))
    inv = np.full(N, (2 ** bits - 1) / 1.5, np.float32)
    g = vt.vitint_linear(x, 1.0, w, dev(s_w), dev(bias), vt.Epilogue(mode=vt.EPI_REQUANT, act=1, inv_out_step=dev(inv), out_bits=bits,
                                                                    out_signed=False, out_container=8))
    _, lo, hi = vo.epilogue_gelu_requant(acc, 1.0, s_w, bias, inv, bits, False, GELU_TOL_REL)
    q = from_codes(g)
    assert ((q >= lo) & (q <= hi)).all() and padding_is_zero(g)


# ---- codes of a width that is no multiple of the column block: one column into a block, around sixteen columns, one short of a
# ---- block, a last tile of several blocks, several tiles a CTA; below a block, and where there is little to do, gemm_i8_kernel
@pytest.mark.parametrize("M,K,N", [(1, 64, 65), (129, 48, 63), (300, 144, 79), (197, 256, 80), (70, 128, 127), (197, 320, 200), (600, 768, 1290),
                                   (5000, 128, 1290), (2600, 64, 2306), (13000, 1000, 65), (5200, 2000, 79), (20100, 320, 127)])
@pytest.mark.parametrize("bits,packed", [(2, False), (4, False), (8, False), (4, True), (2, True)])
def test_linear_codes_of_ragged_width(M, K, N, bits, packed):
    qx, qw = rand_codes(121 + M, (M, K), bits, True), rand_codes(122 + N, (N, K), bits, True)
    form = to_codes if packed else byte_codes
    x, w = form(qx, bits, True), form(qw, bits, True)
    acc = vo.matmul_i32(qx, qw)
    s_w = ((np.abs(si.normal(123, (N,), 0.0, 0.2)) + 0.5) / max(float(np.abs(acc).mean()), 1.0)).astype(np.float32)
    bias = si.normal(124, (N,), 0.0, 0.3)
    alpha = s_w * np.float32(2 ** (bits - 1))
    for cont, pitch in ((8, None), (0, None), (8, (N + 15) // 16 * 16 + 48)):
        out = vt.Codes.empty(M, N, bits, True, container=cont, pitch=pitch)
        out.data.fill_(0xA5)
        vt.vitint_linear(x, 1.0, w, None, None, vt.Epilogue(mode=vt.EPI_REQUANT, alpha=dev(alpha), beta=dev(bias), out_bits=bits,
                                                            out_signed=True, out_container=cont), out=out)
        assert np.array_equal(from_codes(out), vo.epilogue_requant(acc, alpha, bias, bits, True)) and padding_is_zero(out)
    inv = np.full(N, (2 ** bits - 1) / 1.5, np.float32)
    g = vt.vitint_linear(x, 1.0, w, dev(s_w), dev(bias), vt.Epilogue(mode=vt.EPI_REQUANT, act=1, inv_out_step=dev(inv), out_bits=bits,
                                                                    out_signed=False, out_container=8))
    _, lo, hi = vo.epilogue_gelu_requant(acc, 1.0, s_w, bias, inv, bits, False, GELU_TOL_REL)
    q = from_codes(g)
    assert ((q >= lo) & (q <= hi)).all() and padding_is_zero(g)


# ---- packed operands, many row tiles: CTAs that keep their columns' expanded weights, with K blocks of one to six, partial last
# ---- K blocks, a ragged last tile of columns; and few row tiles, which expand as they go
@pytest.mark.parametrize("M,K,N", [(300, 256, 576), (9000, 64, 576), (14001, 200, 192), (20000, 640, 200), (14000, 768, 384), (20000, 96, 1152)])
@pytest.mark.parametrize("bits", [2, 3, 4])
def test_linear_packed_many_rows(M, K, N, bits):
    qx, qw = rand_codes(131 + M, (M, K), bits, True), rand_codes(132 + N, (N, K), bits, True)
    x, w, acc = to_codes(qx, bits, True), to_codes(qw, bits, True), vo.matmul_i32(qx, qw)
    s_w = ((np.abs(si.normal(133, (N,), 0.0, 0.2)) + 0.5) / max(float(np.abs(acc).mean()), 1.0)).astype(np.float32)
    bias, alpha = si.normal(134, (N,), 0.0, 0.3), s_w * np.float32(2 ** (bits - 1))
    out = vt.vitint_linear(x, 1.0, w, None, None, vt.Epilogue(mode=vt.EPI_REQUANT, alpha=dev(alpha), beta=dev(bias), out_bits=bits, out_signed=True))
    assert np.array_equal(from_codes(out), vo.epilogue_requant(acc, alpha, bias, bits, True)) and padding_is_zero(out)
    y = vt.vitint_linear(x, 0.75, w, dev(s_w), dev(bias), vt.Epilogue(mode=vt.EPI_DEQUANT_F32))
    assert np.array_equal(y.cpu().numpy().view(np.uint32), vo.epilogue_dequant(acc, np.float32(0.75), s_w, bias, None).view(np.uint32))


@pytest.mark.parametrize("M,K,N,bits", [(14001, 200, 192, 4), (20000, 96, 1152, 2), (14000, 640, 384, 3)])
def test_linear_packed_many_rows_with_a_residual(M, K, N, bits):
    """Kept weights beside a residual that is read ahead; the residual may be the output buffer."""
    qx, qw = rand_codes(141 + M, (M, K), bits, True), rand_codes(142 + N, (N, K), bits, True)
    acc = vo.matmul_i32(qx, qw)
    s_w, bias, res = (np.abs(si.normal(143, (N,), 0.0, 0.02)) + 1e-3).astype(np.float32), si.normal(144, (N,), 0.0, 0.3), si.normal(145, (M, N))
    want = vo.epilogue_dequant(acc, np.float32(0.75), s_w, bias, res).view(np.uint32)
    x, w = to_codes(qx, bits, True), to_codes(qw, bits, True)
    r = dev(res)
    epi = vt.Epilogue(mode=vt.EPI_DEQUANT_F32, residual=r)
    assert np.array_equal(vt.vitint_linear(x, 0.75, w, dev(s_w), dev(bias), epi).cpu().numpy().view(np.uint32), want)
    vt.vitint_linear(x, 0.75, w, dev(s_w), dev(bias), epi, out=r)
    assert np.array_equal(r.cpu().numpy().view(np.uint32), want)


@pytest.mark.parametrize("M,N", [(16300, 768), (16250, 768)])
def test_linear_fp32_dispatch_boundary(M, N):
    """Around the size from which a short contraction with a residual takes the staged fp32 epilogue."""
    K = 96
    qx, qw = rand_codes(111, (M, K), 4, True), rand_codes(112, (N, K), 4, True)
    s_w = (np.abs(si.normal(113, (N,), 0.0, 0.01)) + 1e-3).astype(np.float32)
    bias, res = si.normal(114, (N,), 0.0, 0.05), si.normal(115, (M, N))
    y = vt.vitint_linear(byte_codes(qx, 4, True), 0.37, byte_codes(qw, 4, True), dev(s_w), dev(bias),
                         vt.Epilogue(mode=vt.EPI_DEQUANT_F32, residual=dev(res)))
    want = vo.epilogue_dequant(vo.matmul_i32(qx, qw), np.float32(0.37), s_w, bias, res)
    assert np.array_equal(y.cpu().numpy().view(np.uint32), want.view(np.uint32))


@pytest.mark.parametrize("M,K,N", [(129, 64, 96), (3000, 128, 768), (25216, 64, 768)])
def test_linear_residual_in_place(M, K, N):
    """out is the residual: several calls in a row on one buffer, as an accumulating caller makes them."""
    qx, qw = rand_codes(151, (M, K), 4, True), rand_codes(152, (N, K), 4, True)
    acc, s_w, y = vo.matmul_i32(qx, qw), np.full(N, np.float32(0.01), np.float32), si.normal(153, (M, N))
    x, w, buf = byte_codes(qx, 4, True), byte_codes(qw, 4, True), dev(y)
    for _ in range(6):
        vt.vitint_linear(x, 0.75, w, dev(s_w), None, vt.Epilogue(mode=vt.EPI_DEQUANT_F32, residual=buf), out=buf)
        y = vo.epilogue_dequant(acc, np.float32(0.75), s_w, None, y)
    assert np.array_equal(buf.cpu().numpy().view(np.uint32), y.view(np.uint32))


# ---- recorded layers: the plan against the same launches one by one ------------------------------------------------
def small_layer(kw, layer=0, cfg=None):
    from paper_2504_18547_b200.encoder import EncoderLayer
    cfg = cfg or si.BlockConfig("plan", 2, kw.pop("tokens", 50), 128, 2, kw.pop("bits", 4), mlp_dim=320)
    return cfg, EncoderLayer(cfg.batch, cfg.tokens, cfg.heads, cfg.mlp_dim, cfg.bits, si.layer_parameters(cfg, layer), **kw)


def one_by_one(layer, x):
    """The layer with an event after every stage: the launches, not the plan."""
    out = torch.empty_like(x)
    layer.forward(x, out, events=[])
    return out


@pytest.mark.parametrize("kw", [{}, {"softmax": "shift", "layernorm": "compare"}, {"bits": 8}, {"fused_attention": False, "bits": 3},
                                {"softmax": "shift", "fused_attention": False}, {"tokens": 300}, {"wide_activations": False, "bits": 2}],
                         ids=lambda kw: "-".join(f"{k}_{v}" for k, v in kw.items()) or "plain")
def test_layer_plan_equals_its_launches(kw):
    cfg, layer = small_layer(dict(kw))
    assert layer._plan is not None
    for i in range(3):                                       # other inputs in other buffers, one of them on another stream
        x = dev(si.normal(300 + i, (cfg.rows, cfg.dim)))
        out = torch.full_like(x, float("nan"))
        stream = torch.cuda.Stream() if i == 1 else torch.cuda.current_stream()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            layer.forward(x, out)
        torch.cuda.synchronize()
        assert torch.equal(out, one_by_one(layer, x))
    # an output whose rows start on 16 bytes only, a strided input, and a replaced parameter
    flat = torch.empty(cfg.rows * cfg.dim + 4, device="cuda")
    odd = flat[4:].view(cfg.rows, cfg.dim)
    layer.forward(x, odd)
    assert torch.equal(odd, out)
    wide = torch.zeros((cfg.rows, cfg.dim + 4), device="cuda")
    wide[:, :cfg.dim] = x
    layer.forward(wide[:, :cfg.dim], odd)
    assert torch.equal(odd, out)
    layer.bias["fc2"] = layer.bias["fc2"] + 1.0
    layer.forward(x, odd)
    assert torch.equal(odd, one_by_one(layer, x)) and not torch.equal(odd, out)


@pytest.mark.parametrize("batch,mlp", [(1, 320), (1, 330), (1, 1024), (3, 2176), (60, 512), (60, 1290)])
def test_plan_sees_weights_written_in_place_right_before_it(batch, mlp):
    """Recorded kernels read weights and parameters ahead of the kernel in front of them, never ahead of the stream: copies into
    the layer's own tensors and runs in turn, nothing between them.  (MLP widths whose weights fill the ring of fc2 and exceed it.)"""
    from paper_2504_18547_b200.encoder import EncoderLayer
    cfg = si.BlockConfig("inplace", batch, 50, 128, 2, 4, mlp_dim=mlp)
    prm, other = si.layer_parameters(cfg, 0), si.layer_parameters(cfg, 1)
    scalars = {k: v for k, v in prm.items() if np.ndim(v) == 0}
    layers = [EncoderLayer(batch, 50, 2, mlp, 4, dict(p, **scalars)) for p in (prm, other)]

    def tensors(layer):
        return ([c.data for c in layer.w.values()] + list(layer.s_w.values()) + list(layer.bias.values())
                + [layer.alpha_qkv, layer.beta_qkv, layer.alpha_o, layer.inv_s_g, layer.ln1_g, layer.ln1_b, layer.ln2_g, layer.ln2_b])
    states = [[t.clone() for t in tensors(layer)] for layer in layers]
    x = dev(si.normal(350 + batch, (cfg.rows, cfg.dim)))
    want = [one_by_one(layer, x) for layer in layers]
    assert not torch.equal(want[0], want[1])
    outs = [torch.empty_like(x) for _ in range(8)]
    torch.cuda.synchronize()
    for i, out in enumerate(outs):
        for t, new in zip(tensors(layers[0]), states[i & 1]):
            t.copy_(new)
        layers[0].forward(x, out)
    assert layers[0]._plan is not None
    for i, out in enumerate(outs):
        assert torch.equal(out, want[i & 1])


@pytest.mark.parametrize("batch", [1, 60, 160])
@pytest.mark.parametrize("packed", [False, True])
def test_plan_sees_an_exp_table_written_in_place_right_before_it(batch, packed):
    """The recorded attention core reads its table ahead of the kernel in front of it, never ahead of the stream: another score
    scale's table and runs in turn, with items for one group of warps in a CTA and for two."""
    from paper_2504_18547_b200.encoder import EncoderLayer
    cfg = si.BlockConfig("table", batch, 50, 128, 2, 4, mlp_dim=320)
    layer = EncoderLayer(batch, 50, 2, 320, 4, si.layer_parameters(cfg), wide_activations=not packed)
    tables = [layer.attn_table.clone(), vt.vitint_attention_exp_table(4, 6 * layer.s_q, layer.s_k)]
    x = dev(si.normal(360 + batch, (cfg.rows, cfg.dim)))
    want = []
    for t in tables:
        layer.attn_table.copy_(t)
        want.append(one_by_one(layer, x))
    assert not torch.equal(want[0], want[1])
    outs = [torch.empty_like(x) for _ in range(8)]
    torch.cuda.synchronize()
    for i, out in enumerate(outs):
        layer.attn_table.copy_(tables[i & 1])
        layer.forward(x, out)
    assert layer._plan is not None
    for i, out in enumerate(outs):
        assert torch.equal(out, want[i & 1])


@pytest.mark.parametrize("kw", [{}, {"fused_attention": False}, {"bits": 8}], ids=["core", "three_kernels", "bits8"])
def test_plan_follows_every_parameter_that_the_launches_read(kw):
    cfg, layer = small_layer(dict(kw))
    x = dev(si.normal(352, (cfg.rows, cfg.dim)))
    seen = []

    def same(changed=True):
        out = layer.forward(x, torch.empty_like(x))
        assert torch.equal(out, one_by_one(layer, x))
        assert not seen or torch.equal(out, seen[-1]) != changed
        seen.append(out)

    same()
    layer.epi_qkv.alpha = layer.epi_qkv.alpha * 0.5
    same()
    layer.epi_qkv.beta = None
    same()
    layer.epi_fc1.inv_out_step = layer.epi_fc1.inv_out_step * 0.5
    same()
    for name in ("proj", "fc1", "fc2"):
        layer.bias[name] = None
        same()
    layer.alpha_qkv, layer.beta_qkv, layer.inv_s_g = (t * 3.0 for t in (layer.alpha_qkv, layer.beta_qkv, layer.inv_s_g))
    same(changed=False)                                     # the launches read the epilogues
    if layer.fused_attention:
        layer.alpha_o = layer.alpha_o * 0.5
        same()
    else:
        layer.epi_o.alpha = layer.epi_o.alpha * 0.5
        same()
        assert layer._plan is not None
        layer.epi_o.beta = torch.full((cfg.dim,), 1.0, device="cuda")      # no recorded layer has it: launched one by one
        same()
        layer.epi_o.beta = None
        same()


@pytest.mark.parametrize("kw", [{}, {"bits": 8}, {"fused_attention": False}, {"softmax": "shift", "layernorm": "compare"}],
                         ids=["core", "bits8", "bounded", "paper"])
def test_layers_and_stacks_can_be_copied_and_pickled(kw):
    import copy
    import pickle
    from paper_2504_18547_b200.encoder import EncoderStack
    cfg, layer = small_layer(dict(kw))
    kw = {k: v for k, v in kw.items() if k != "bits"}
    stack = EncoderStack([si.layer_parameters(cfg, l) for l in range(3)], cfg.batch, cfg.tokens, cfg.heads, cfg.mlp_dim, cfg.bits, **kw)
    x = dev(si.normal(350, (cfg.rows, cfg.dim)))
    for m in (layer, stack):
        want = m.forward(x, torch.empty_like(x))
        for other in (copy.deepcopy(m), copy.copy(m), pickle.loads(pickle.dumps(m))):
            assert torch.equal(other.forward(x, torch.empty_like(x)), want)
            assert other._plan is not None and other._plan is not m._plan
        del other
        assert torch.equal(m.forward(x, torch.empty_like(x)), want)


def test_stack_without_a_plan():
    from paper_2504_18547_b200.encoder import EncoderStack
    cfg = si.BlockConfig("plan", 1, 40, 64, 1, 4, mlp_dim=128)
    stacks = [EncoderStack([si.layer_parameters(cfg, l) for l in range(2)], 1, 40, 1, 128, 4, plan=plan) for plan in (True, False)]
    x = dev(si.normal(353, (40, 64)))
    a, b = (s.forward(x, torch.empty_like(x)) for s in stacks)
    assert torch.equal(a, b) and stacks[0]._plan is not None and stacks[1]._plan is None


def test_plan_comes_back_with_the_parameter_that_was_refused():
    from paper_2504_18547_b200.encoder import EncoderStack
    cfg, layer = small_layer({})
    stack = EncoderStack([si.layer_parameters(cfg, l) for l in range(2)], cfg.batch, cfg.tokens, cfg.heads, cfg.mlp_dim, cfg.bits)
    x = dev(si.normal(351, (cfg.rows, cfg.dim)))
    for m, part in ((layer, layer), (stack, stack.layers[1])):
        want = m.forward(x, torch.empty_like(x))
        good, part.s_p = part.s_p, -1.0
        with pytest.raises(vt.VitintError):
            m.forward(x, torch.empty_like(x))
        assert m._plan is None
        part.s_p = good
        assert torch.equal(m.forward(x, torch.empty_like(x)), want) and m._plan is not None


@pytest.mark.parametrize("kw", [{}, {"softmax": "shift"}, {"fused_attention": False, "bits": 8}, {"fused_attention": False},
                                {"softmax": "shift", "fused_attention": False}, {"bits": 8}],
                         ids=["exp_core", "shift_core", "exp", "exp_bounded", "shift", "exp_core_any"])
def test_encoder_forward_equals_the_plan(kw):
    """vitint_encoder_forward for every kind of attention, on one and three layers, the table of the bounded softmax not filled."""
    import ctypes
    from paper_2504_18547_b200 import binding as B
    from paper_2504_18547_b200.encoder import EncoderStack
    kw = dict(kw)
    cfg = si.BlockConfig("forward", 2, 50, 128, 2, kw.pop("bits", 4), mlp_dim=320)
    x = dev(si.normal(330, (cfg.rows, cfg.dim)))
    for n in (1, 3):
        stack = EncoderStack([si.layer_parameters(cfg, l) for l in range(n)], cfg.batch, cfg.tokens, cfg.heads, cfg.mlp_dim, cfg.bits, **kw)
        want, out = stack.forward(x, torch.empty_like(x)), torch.full_like(x, float("nan"))
        assert stack._plan is not None
        for l in stack.layers:
            if getattr(l, "sm_table", None) is not None:
                l.sm_table.zero_()
        descs, bufs = (B._EncoderLayerDesc * n)(*[l._desc() for l in stack.layers]), (ctypes.c_void_p * 2)(*[b.data_ptr() for b in stack.buf])
        assert B.lib().vitint_encoder_forward(descs, n, bufs, x.data_ptr(), out.data_ptr(), B._stream()) == 0
        assert torch.equal(out, want)


def test_layer_plan_inside_a_captured_graph():
    cfg, layer = small_layer({})
    x, out = dev(si.normal(310, (cfg.rows, cfg.dim))), torch.empty((cfg.rows, cfg.dim), device="cuda")
    layer.forward(x, out)
    want = out.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        layer.forward(x, out)
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)


@pytest.mark.parametrize("replay_first", [True, False])
@pytest.mark.parametrize("plan", [True, False])
@pytest.mark.parametrize("kw", [{}, {"fused_attention": False}], ids=["core", "bounded"])
def test_layer_changed_during_a_capture(kw, plan, replay_first):
    """A parameter replaced inside a capture: the captured launches, and eager ones before the graph has run once or after it."""
    (cfg, layer), (_, fresh) = small_layer(dict(kw, plan=plan)), small_layer(dict(kw, plan=False))
    x = dev(si.normal(370, (cfg.rows, cfg.dim)))
    if plan:
        layer.forward(x, torch.empty_like(x))
    fresh.bias["fc2"] = bias = layer.bias["fc2"] + 1.0
    fresh.c = c = float(np.float32(layer.c * 0.5)) if kw else layer.c
    want = fresh.forward(x, torch.empty_like(x))
    out, eager, graph = torch.zeros_like(x), torch.zeros_like(x), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        layer.bias["fc2"], layer.c = bias, c
        layer.forward(x, out)
    if replay_first:
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
    layer.forward(x, eager)
    assert torch.equal(eager, want) and (layer._plan is not None) == plan
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)


def test_plans_made_run_and_dropped_during_a_capture():
    """Neither the capturing thread's plans nor another thread's forward() may end a capture."""
    import threading
    from paper_2504_18547_b200 import binding as B
    cfg, layer = small_layer({})
    (_, other), (_, dropped) = small_layer({}), small_layer({})
    x = dev(si.normal(312, (cfg.rows, cfg.dim)))
    out, elsewhere, late = (torch.zeros_like(x) for _ in range(3))
    want = layer.forward(x, torch.empty_like(x)).clone()
    stream, errors = torch.cuda.Stream(), []
    torch.cuda.synchronize()

    def beside():
        try:
            with torch.cuda.stream(stream):
                other.forward(x, elsewhere)
        except Exception as e:                               # noqa: BLE001 -- reported by the main thread
            errors.append(e)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        layer.forward(x, out)
        del dropped
        plan = B.EncoderPlan([layer._desc()])
        t = threading.Thread(target=beside)
        t.start()
        t.join()
    assert not errors
    graph.replay()
    plan.run(x, late)
    torch.cuda.synchronize()
    assert torch.equal(out, want) and torch.equal(elsewhere, want) and torch.equal(late, want)


def test_stack_plan_from_two_threads():
    import threading
    from paper_2504_18547_b200.encoder import EncoderStack
    cfg = si.BlockConfig("plan", 1, 40, 64, 1, 4, mlp_dim=128)
    stacks = [EncoderStack([si.layer_parameters(cfg, l + 5 * k) for l in range(3)], 1, 40, 1, 128, 4) for k in range(2)]
    xs = [dev(si.normal(320 + i, (40, 64))) for i in range(6)]
    want = [[], []]
    for k, st in enumerate(stacks):
        for x in xs:
            cur = x
            for l in st.layers:
                cur = one_by_one(l, cur)
            want[k].append(cur)
    torch.cuda.synchronize()
    got, errors = [[], []], []

    def work(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for x in xs:
                    got[k].append(stacks[k].forward(x, torch.empty_like(x)))
                torch.cuda.current_stream().synchronize()
        except Exception as e:                               # noqa: BLE001 -- reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    [t.start() for t in threads]
    [t.join() for t in threads]
    assert not errors
    for k in range(2):
        for a, b in zip(got[k], want[k]):
            assert torch.equal(a, b)


def test_one_plan_from_two_threads():
    """Two threads run ONE plan with their own x and out on one stream: rewriting the nodes and launching are one step."""
    import threading
    cfg, layer = small_layer({})
    xs = [dev(si.normal(360 + i, (cfg.rows, cfg.dim))) for i in range(8)]
    want = [one_by_one(layer, x) for x in xs]
    stream, errors, got, start = torch.cuda.Stream(), [], [[], []], threading.Barrier(2)
    outs = [[torch.empty_like(xs[0]) for _ in range(200)] for _ in range(2)]
    torch.cuda.synchronize()

    def work(k):
        try:
            with torch.cuda.stream(stream):
                start.wait()
                for i, out in enumerate(outs[k]):
                    got[k].append((layer.forward(xs[(i + 3 * k) % 8], out), (i + 3 * k) % 8))
        except Exception as e:                               # noqa: BLE001 -- reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    [t.start() for t in threads]
    [t.join() for t in threads]
    torch.cuda.synchronize()
    assert not errors and layer._plan is not None
    assert all(torch.equal(out, want[i]) for k in range(2) for out, i in got[k])


@pytest.mark.parametrize("bits", [2, 4])
def test_shift_core_limit_of_the_logits(bits):
    """64 m^2 c log2(e) <= 30000: taken right below, refused right above."""
    heads, tokens, D, m = 1, 9, 64, 2 if bits == 2 else 8
    codes, alpha = byte_codes(rand_codes(541, (tokens, 3 * D), bits, True), bits, True), torch.ones(D, device="cuda")
    step = (30000.0 / (64 * m * m * np.log2(np.e)) * 8) ** 0.5
    vt.vitint_attention_core_shift(codes, 1, heads, tokens, 0.999 * step, step, 0.05, bits, alpha, None)
    with pytest.raises(vt.VitintError) as e:
        vt.vitint_attention_core_shift(codes, 1, heads, tokens, 1.001 * step, step, 0.05, bits, alpha, None)
    assert e.value.code == -2


# ---- bit-packed operands: both packed alike (the reordered unpacking), packed unlike, one of them byte-stored; K at the
# ---- edges of a 32-code MMA step, a 64-code chunk and a 128-code block
@pytest.mark.parametrize("M,K,N", [(1, 16, 64), (33, 33, 64), (129, 96, 128), (130, 200, 192), (197, 1000, 320), (2000, 160, 1152)])
@pytest.mark.parametrize("bx,bw", [(4, 4), (2, 2), (3, 4), (2, 4), (4, 2)])
@pytest.mark.parametrize("xs", [True, False])
def test_linear_packed_operands(M, K, N, bx, bw, xs):
    qx, qw = rand_codes(121 + M, (M, K), bx, xs), rand_codes(122 + N, (N, K), bw, True)
    acc = vo.matmul_i32(qx, qw)
    spread = max(float(np.abs(acc).mean()), 1.0)
    alpha = ((np.abs(si.normal(123, (N,), 0.0, 0.2)) + 0.5) * 2 / spread).astype(np.float32)
    beta, res = si.normal(124, (N,), 0.0, 0.3), si.normal(125, (M, N))
    px, pw = to_codes(qx, bx, xs), to_codes(qw, bw, True)
    for x, w in ((px, pw), (px, vt.vitint_widen(pw)), (vt.vitint_widen(px), pw)):
        q = vt.vitint_linear(x, 1.0, w, None, None, vt.Epilogue(mode=vt.EPI_REQUANT, alpha=dev(alpha), beta=dev(beta), out_bits=4,
                                                                out_signed=True))
        assert np.array_equal(from_codes(q), vo.epilogue_requant(acc, alpha, beta, 4, True)) and padding_is_zero(q)
        y = vt.vitint_linear(x, 0.75, w, dev(alpha), dev(beta), vt.Epilogue(mode=vt.EPI_DEQUANT_F32, residual=dev(res)))
        want = vo.epilogue_dequant(acc, np.float32(0.75), alpha, beta, res)
        assert np.array_equal(y.cpu().numpy().view(np.uint32), want.view(np.uint32))


def test_linear_packed_large_sums():
    """Sums beyond 2^22 (converted with their power-of-two scale) and the largest the packed path takes."""
    M, K, N = 130, 8000, 64
    qx, qw = np.full((M, K), -8, np.int16), rand_codes(131, (N, K), 4, True)
    qw[0], qw[1] = -8, 7
    acc = vo.matmul_i32(qx, qw)
    s_w = np.full(N, 1e-4, np.float32)
    y = vt.vitint_linear(to_codes(qx, 4, True), 0.75, to_codes(qw, 4, True), dev(s_w), None, vt.Epilogue(mode=vt.EPI_DEQUANT_F32))
    want = vo.epilogue_dequant(acc, np.float32(0.75), s_w)
    assert np.array_equal(y.cpu().numpy().view(np.uint32), want.view(np.uint32))
    K = 70000                                               # 70000 * 64 > 2^22
    qx, qw = rand_codes(132, (M, K), 4, True), rand_codes(133, (N, K), 4, True)
    qx[0], qw[0] = -8, -8
    y = vt.vitint_linear(to_codes(qx, 4, True), 0.75, to_codes(qw, 4, True), dev(s_w), None, vt.Epilogue(mode=vt.EPI_DEQUANT_F32))
    want = vo.epilogue_dequant(vo.matmul_i32(qx, qw), np.float32(0.75), s_w)
    assert np.array_equal(y.cpu().numpy().view(np.uint32), want.view(np.uint32))


# ---- sizes whose packed ring has three slots (the launcher's arithmetic: 224 columns of fp32 output or 192 of the norm kind with
# ---- both operands packed, 256 columns with one of them byte-stored or 2-bit), many K blocks, several tiles a CTA
@pytest.mark.parametrize("M,K,N,bx,bw,kind", [(4000, 1100, 896, 4, 4, "fp32"), (12608, 896, 896, 4, 4, "fp32"), (4000, 1100, 896, 2, 4, "fp32"),
                                              (4000, 1100, 1024, 8, 4, "codes"), (4000, 1100, 1024, 4, 2, "codes"),
                                              (2000, 1100, 1344, 4, 4, "norm")])
def test_linear_packed_three_slot_ring(M, K, N, bx, bw, kind):
    qx, qw = rand_codes(141, (M, K), bx, True), rand_codes(142, (N, K), bw, True)
    acc = vo.matmul_i32(qx, qw)
    spread = max(float(np.abs(acc).mean()), 1.0)
    alpha = ((np.abs(si.normal(143, (N,), 0.0, 0.2)) + 0.5) * 2 / spread).astype(np.float32)
    beta = si.normal(144, (N,), 0.0, 0.3)
    x, w = to_codes(qx, bx, True), to_codes(qw, bw, True)
    for _ in range(5):                                      # the order in which copies land differs from run to run
        if kind == "codes":
            q = vt.vitint_linear(x, 1.0, w, None, None, vt.Epilogue(mode=vt.EPI_REQUANT, alpha=dev(alpha), beta=dev(beta), out_bits=4,
                                                                    out_signed=True))
            assert np.array_equal(from_codes(q), vo.epilogue_requant(acc, alpha, beta, 4, True))
        elif kind == "fp32":
            y = vt.vitint_linear(x, 0.75, w, dev(alpha), dev(beta), vt.Epilogue(mode=vt.EPI_DEQUANT_F32))
            want = vo.epilogue_dequant(acc, np.float32(0.75), alpha, beta)
            assert np.array_equal(y.cpu().numpy().view(np.uint32), want.view(np.uint32))
        else:
            D = N // 3
            rf = [compare_case(2, 64, 4, 480 + k) for k in range(2)]
            refs, flips, n_eps = [r for _, r, _, _ in rf], [f for _, _, f, _ in rf], rf[0][3]
            got, _ = vt.vitint_linear_qkv_norm(x, 0.5, w, dev(alpha), dev(beta), dev(np.stack(refs)), dev(np.stack(flips)), n_eps,
                                               dev(alpha[2 * D:]), dev(beta[2 * D:]), 4)
            y = vo.epilogue_dequant(acc, np.float32(0.5), alpha, beta)
            want = [compare_reference(y[:, k * D:(k + 1) * D].reshape(M * D // 64, 64), refs[k], flips[k], n_eps, 4).reshape(M, D)
                    for k in range(2)] + [vo.epilogue_requant(acc[:, 2 * D:], alpha[2 * D:], beta[2 * D:], 4, True)]
            assert np.array_equal(from_codes(got), np.concatenate(want, axis=1))


# ---- comparator LayerNorm: column slabs, staged chunks and rounds of rows; references no uniform quantizer would give ------
def compare_case(rows, cols, bits, seed, refs=None):
    x = si.normal(seed, (rows, cols), 0.3, 1.7)
    g, b = si.normal(seed + 1, (cols,), 1.0, 0.02), si.normal(seed + 2, (cols,), 0.0, 0.02)
    g[::3] *= -1
    step = si.gaussian_lsq_step(1.0, bits)
    n_eps = float(np.float32(np.float64(cols) * np.float64(np.float32(1e-6))))
    r, f = vt.fold_layernorm_references(g, b, step, bits, True, cols)
    return x, (r if refs is None else refs(r)), f, n_eps


def compare_reference(x, refs, flip, n_eps, bits):
    """The definition: Eq. 5 in fp32, then the count of references exceeded."""
    mu, s = np.zeros(x.shape[0], np.float32), np.zeros(x.shape[0], np.float32)
    for i in range(x.shape[1]):
        delta = x[:, i] - mu
        mu = mu + delta / np.float32(i + 1)
        s = s + delta * (x[:, i] - mu)
    v = s + np.float32(n_eps)
    d = (x - mu[:, None]) * np.where(flip, np.float32(-1), np.float32(1))
    ds = np.copysign(d * d, d)
    cnt = np.zeros(x.shape, np.int16)
    with np.errstate(invalid="ignore"):
        for t in range(refs.shape[1]):
            cnt += ds > v[:, None] * refs[:, t]
    return cnt - (1 << (bits - 1))


@pytest.mark.parametrize("rows,cols", [(1, 4), (7, 64), (33, 68), (300, 772), (149, 1540), (28500, 64)])
@pytest.mark.parametrize("bits,cont", [(2, 0), (3, 8), (4, 0), (4, 8)])
def test_compare_layernorm_tiling(rows, cols, bits, cont):
    x, refs, flip, n_eps = compare_case(rows, cols, bits, 400 + cols)
    out = vt.Codes.empty(rows, cols, bits, True, container=cont)
    out.data.fill_(0xA5)
    got, _ = vt.vitint_layernorm_compare_quantize(dev(x), dev(refs), dev(flip), n_eps, bits, True, out=out)
    assert np.array_equal(from_codes(got), compare_reference(x, refs, flip, n_eps, bits)) and padding_is_zero(got)


@pytest.mark.parametrize("warp", ["squeezed", "equal", "huge"])
def test_compare_layernorm_references_that_are_not_uniform(warp):
    """Ascending references for which the count cannot be guessed: it is found all the same."""
    def refs(r):
        if warp == "equal":
            return np.repeat(r[:, 7:8], r.shape[1], axis=1)
        if warp == "huge":
            return np.sort(r * np.float32(1e30), axis=1)
        return np.sort((np.sign(r) * np.abs(r) ** 3 * 1e3).astype(np.float32), axis=1)
    x, refs_, flip, n_eps = compare_case(90, 256, 4, 450, refs)
    got, _ = vt.vitint_layernorm_compare_quantize(dev(x), dev(refs_), dev(flip), n_eps, 4, True)
    assert np.array_equal(from_codes(got), compare_reference(x, refs_, flip, n_eps, 4))


@pytest.mark.parametrize("M,heads,bits", [(1, 1, 2), (129, 3, 4), (300, 5, 3), (2000, 7, 4), (2600, 7, 3), (6500, 7, 4)])
@pytest.mark.parametrize("packed", [False, True])
def test_qkv_norm_tiles_and_references(M, heads, bits, packed):
    """Segments that end inside a tile, packed operands, one to four tiles a CTA, and references no uniform quantizer would give."""
    D, K = 64 * heads, 96
    qx, qw = rand_codes(461, (M, K), bits, True), rand_codes(462, (3 * D, K), bits, True)
    acc = vo.matmul_i32(qx, qw)
    s_w = (np.abs(si.normal(463, (3 * D,), 0.0, 0.01)) + 1e-3).astype(np.float32)
    bias = si.normal(464, (3 * D,), 0.0, 0.05)
    y = vo.epilogue_dequant(acc, np.float32(0.5), s_w, bias)
    rf = [compare_case(2, 64, bits, 470 + k) for k in range(2)]
    n_eps = rf[0][3]
    alpha, beta = np.full(D, 0.3, np.float32), si.normal(465, (D,), 0.0, 0.3)
    x, w = to_codes(qx, bits, True), to_codes(qw, bits, True)
    if not packed:
        x, w = byte_codes(qx, bits, True), byte_codes(qw, bits, True)
    for odd in (False, True):
        refs = [np.sort((np.sign(r) * np.abs(r) ** 3 * 1e3).astype(np.float32), axis=1) if odd else r for _, r, _, _ in rf]
        flips = [f for _, _, f, _ in rf]
        got, _ = vt.vitint_linear_qkv_norm(x, 0.5, w, dev(s_w), dev(bias), dev(np.stack(refs)), dev(np.stack(flips)), n_eps,
                                           dev(alpha), dev(beta), bits)
        want = [compare_reference(y[:, k * D:(k + 1) * D].reshape(M * heads, 64), refs[k], flips[k], n_eps, bits).reshape(M, D)
                for k in range(2)] + [vo.epilogue_requant(acc[:, 2 * D:], alpha, beta, bits, True)]
        assert np.array_equal(from_codes(got), np.concatenate(want, axis=1)) and padding_is_zero(got)


@pytest.mark.parametrize("M,heads,bits", [(1, 1, 3), (130, 3, 3), (2600, 7, 4), (6500, 7, 3), (12000, 4, 2)])
def test_qkv_norm_statistics_and_codes_of_both_groups(M, heads, bits):
    """No second tile in a CTA (the second group of epilogue warps has none), then one to six tiles: every Q and K head's
    statistics, and its codes, which read tables that all groups share."""
    D, K = 64 * heads, 64
    qx, qw = rand_codes(481 + M, (M, K), bits, True), rand_codes(482, (3 * D, K), bits, True)
    s_w = (np.abs(si.normal(483, (3 * D,), 0.0, 0.01)) + 1e-3).astype(np.float32)
    bias = si.normal(484, (3 * D,), 0.0, 0.05)
    y = vo.epilogue_dequant(vo.matmul_i32(qx, qw), np.float32(0.5), s_w, bias)
    rf = [compare_case(2, 64, bits, 490 + k) for k in range(2)]
    got, stats = vt.vitint_linear_qkv_norm(byte_codes(qx, bits, True), 0.5, byte_codes(qw, bits, True), dev(s_w), dev(bias),
                                           dev(np.stack([r for _, r, _, _ in rf])), dev(np.stack([f for _, _, f, _ in rf])), rf[0][3],
                                           dev(np.full(D, 0.3, np.float32)), None, bits)
    codes, stats = from_codes(got), stats.cpu().numpy()
    for k, (_, r, f, n_eps) in enumerate(rf):
        x = y[:, k * D:(k + 1) * D].reshape(M * heads, 64)
        assert np.array_equal(codes[:, k * D:(k + 1) * D].reshape(M * heads, 64), compare_reference(x, r, f, n_eps, bits))
        mu, s = np.zeros(len(x), np.float32), np.zeros(len(x), np.float32)
        for i in range(64):
            delta = x[:, i] - mu
            mu = mu + delta / np.float32(i + 1)
            s = s + delta * (x[:, i] - mu)
        assert np.array_equal(stats[k, :, 0].view(np.uint32), mu.view(np.uint32))
        assert np.array_equal(stats[k, :, 1].view(np.uint32), (s + np.float32(n_eps)).view(np.uint32))


# ---- fused attention core: every remainder of the column walk, a quantizer step whose unclamped codes exceed 16 bits -------
@pytest.mark.parametrize("tokens", [1, 7, 8, 9, 31, 33, 63, 64, 72, 128, 129, 160, 192, 200, 225, 255, 256, 257, 320, 415])
@pytest.mark.parametrize("bits,p_scale", [(4, 1.0), (2, 1.0), (4, 1e-5)])
def test_attention_core_column_walk(tokens, bits, p_scale):
    """Against the oracle's Q K^T, softmax band and P V: O inside the interval that the band of P reaches."""
    from oracle import pipeline as vp
    batch, heads = 2, 2
    D, n = 64 * heads, batch * heads
    qkv = rand_codes(500 + tokens, (batch * tokens, 3 * D), bits, True)
    s_q = np.float32(0.25 if bits == 4 else 0.75)
    s_p = np.float32(p_scale * 2.0 / (tokens * np.sqrt(2 ** bits - 1)))
    q, k, v = (vp.split_heads(qkv, batch, tokens, heads, 64, i * D) for i in range(3))
    S = vo.qk(q, k)
    _, pc, plo, phi = vo.softmax_quantize(S.reshape(n * tokens, tokens), vp.softmax_scale(s_q, s_q, 64), s_p, bits)
    if p_scale != 1.0:
        assert (pc == 2 ** bits - 1).mean() > 0.5                          # codes far beyond the clamp
    alpha, beta = np.full(D, np.float32(0.05 / tokens ** 0.5), np.float32), si.normal(501, (D,), 0.0, 0.5)
    want = []
    for a, b in ((plo, phi), (phi, plo)):
        acc = vo.pv(a.reshape(n, tokens, tokens), np.maximum(v, 0)) + vo.pv(b.reshape(n, tokens, tokens), np.minimum(v, 0))
        want.append(vo.epilogue_requant(vp.merge_heads(acc, batch, tokens, heads, 64), alpha, beta, bits, True))
    got = vt.vitint_attention_core(byte_codes(qkv, bits, True), batch, heads, tokens, float(s_q), float(s_q), float(s_p), bits,
                                   dev(alpha), dev(beta))
    o = from_codes(got)
    assert ((o >= want[0]) & (o <= want[1])).all() and padding_is_zero(got)


@pytest.mark.parametrize("tokens,bits", [(2056, 4), (2057, 4), (2400, 4), (4096, 4), (4096, 2)])
def test_long_attention_sums_beyond_22_bits(tokens, bits):
    """8-bit P saturated over thousands of tokens, where |O| passes 2^22: all scores equal, so every code of P is 255 and
    O = 255 T v."""
    D = 64
    lo, hi = si.code_range(bits, True)
    qkv = np.zeros((tokens, 3 * D), np.int16)
    qkv[:, 2 * D:] = v = (np.arange(D) % (hi - lo + 1) + lo).astype(np.int16)
    acc = np.broadcast_to((255 * tokens * v.astype(np.int64)).astype(np.int32), (tokens, D)).copy()
    alpha, beta = np.full(D, np.float32(100.0 / (255.0 * 8 * tokens)), np.float32), np.linspace(-20, 20, D).astype(np.float32)
    out = vt.Codes.empty(tokens, D, 8, True)
    vt.vitint_attention_core(byte_codes(qkv, bits, True), 1, 1, tokens, 0.25, 0.25, 1.0 / (300.0 * tokens), 8, dev(alpha), dev(beta),
                             out=out)
    assert np.array_equal(from_codes(out), vo.epilogue_requant(acc, alpha, beta, 8, True))


@pytest.mark.parametrize("tokens", [1, 9, 33, 100, 145, 197, 224, 256])
def test_layer_8bit_core_equals_three_kernels(tokens):
    """8-bit layers: the recorded pass evaluates exp inside the fused core, the launches go through S and P in memory."""
    cfg, layer = small_layer({"bits": 8, "tokens": tokens})
    x = dev(si.normal(600 + tokens, (cfg.rows, cfg.dim)))
    out = torch.empty_like(x)
    layer.forward(x, out)
    o = layer.O.data.clone()
    assert torch.equal(out, one_by_one(layer, x)) and torch.equal(o, layer.O.data)


@pytest.mark.parametrize("tokens", [9, 197])
def test_8bit_layer_keeps_scores_that_are_asked_for(tokens):
    """S and P hold the last call's scores and codes whenever they are looked at; held references follow later calls."""
    cfg, layer = small_layer({"bits": 8, "tokens": tokens})
    _, three = small_layer({"bits": 8, "tokens": tokens, "fused_attention": False})
    assert not hasattr(layer, "no_such_attribute")
    for i in range(4):
        x = dev(si.normal(620 + i, (cfg.rows, cfg.dim)))
        out, want = torch.empty_like(x), torch.empty_like(x)
        layer.forward(x, out) if i != 3 else layer.forward(x, out, events=[])
        three.forward(x, want)
        assert torch.equal(out, want) and layer._plan is not None
        if i == 1:
            S, P = layer.S, layer.P
        if i:
            assert torch.equal(S[:, :tokens], three.S[:, :tokens]) and torch.equal(P.data, three.P.data)


@pytest.mark.parametrize("tokens", [5, 197])
def test_attention_block_8bit_core(tokens):
    """vitint_attention_block with 8-bit codes: with a copy of P (three kernels) and without (the fused core)."""
    cfg = si.BlockConfig("b8", 2, tokens, 128, 2, 8)
    prm = si.layer_parameters(cfg)
    xq = vt.vitint_quantize(dev(si.activations(cfg)), float(prm["s_x"]), 8, True)
    w = {n: vt.vitint_quantize(dev(prm["w_" + n]), 0.0, 8, True, row_steps=dev(prm["s_w_" + n])) for n in ("qkv", "proj")}
    seg = np.repeat(np.array([prm["s_q"], prm["s_k"], prm["s_v"]], np.float32), cfg.dim)
    alpha, beta = vt.fold_requant(prm["s_x"], prm["s_w_qkv"], prm["b_qkv"], seg)
    alpha_o, _ = vt.fold_requant(prm["s_p"], np.full(cfg.dim, prm["s_v"], np.float32), None, prm["s_o"])
    a = vt.AttentionWeights(cfg.batch, tokens, cfg.heads, 8, w["qkv"], dev(alpha), dev(beta), float(prm["s_q"]), float(prm["s_k"]),
                            float(prm["s_v"]), float(prm["s_p"]), float(prm["s_o"]), 8, dev(alpha_o), None, w["proj"],
                            dev(prm["s_w_proj"]), dev(prm["b_proj"]), vt.Epilogue(mode=vt.EPI_DEQUANT_F32))
    p = vt.Codes.empty(cfg.batch * cfg.heads * tokens, tokens, 8, False)
    want = vt.vitint_attention_block(xq, a, dbg_p=p)
    assert torch.equal(vt.vitint_attention_block(xq, a), want)


@pytest.mark.parametrize("tokens", [1, 8, 9, 33, 40, 129, 197, 256])
@pytest.mark.parametrize("bits,p_bits", [(4, 4), (4, 8), (2, 2)])
def test_shift_core_equals_three_kernels(tokens, bits, p_bits):
    """Eq. 4 inside the fused core: rows whose scores lie within a few octaves (summed in doubles), rows spread over hundreds
    (64-bit integers, terms shifted out) and rows of equal scores, whose quantizer arguments sit on ties when T p_step 2 = 1."""
    batch, heads, D = 2, 2, 128
    rng = np.random.default_rng(900 + tokens + bits)
    lo, hi = si.code_range(bits, True)
    qkv = rng.integers(lo, hi + 1, (batch * tokens, 3 * D)).astype(np.int16)
    qkv[::3, :D] //= 2                                    # narrow rows beside wide ones; image 1 mixes them in every warp
    qkv[1::5, :D] = 0                                     # equal scores
    packed = to_codes(qkv, bits, True)
    codes = vt.vitint_widen(packed)
    slabs = [vt.Slabs.of_qkv(packed, tokens, D, i) for i in range(3)]
    alpha = dev(rng.uniform(0.01, 0.05, D).astype(np.float32))
    for scale in (0.02, 0.3, 1.5):
        for p_step in (np.float32(2.0 / tokens / (2 ** p_bits - 1) ** 0.5), np.float32(2.0 / tokens)):
            step = np.float32(scale * 4.0 / (hi + 1))
            c2 = np.float32(np.float64(vp.softmax_scale(step, step, 64)) * np.log2(np.e))
            S = vt.vitint_qk(slabs[0], slabs[1], batch, heads, tokens)
            P = vt.vitint_softmax_shift_quantize(S.view(batch * heads * tokens, -1), tokens, c2, p_step, p_bits)
            epi = vt.Epilogue(mode=vt.EPI_REQUANT, alpha=alpha, out_bits=8, out_signed=True)
            want = from_codes(vt.vitint_pv(P, slabs[2], batch, heads, tokens, 1.0, 1.0, epi))
            out = vt.Codes.empty(batch * tokens, D, 8, True)
            got = from_codes(vt.vitint_attention_core_shift(codes, batch, heads, tokens, step, step, p_step, p_bits, alpha, None,
                                                            out=out))
            assert np.array_equal(got, want), (scale, p_step)


@pytest.mark.parametrize("tokens", [1, 9, 40, 197])
@pytest.mark.parametrize("p_step", [1e-6, 2.0 ** -16, 1.0 / 64999.0, "tie"])
def test_cores_with_codes_on_or_far_beyond_the_last_level(tokens, p_step):
    """Codes proven by an interval around the reciprocal, against the three kernels: steps whose unclamped codes need more than 16
    bits (nothing is proven, every code by comparisons or division) and a step that puts equal probabilities on a tie."""
    step_p = np.float32(2.0 / tokens if p_step == "tie" else p_step)
    batch, heads, D, bits = 1, 2, 128, 4
    qkv = rand_codes(950 + tokens, (batch * tokens, 3 * D), bits, True)
    qkv[::2, :D] = 0                                      # equal scores
    packed = to_codes(qkv, bits, True)
    slabs = [vt.Slabs.of_qkv(packed, tokens, D, i) for i in range(3)]
    alpha, step = dev(np.full(D, np.float32(0.02))), np.float32(0.3)
    c2 = np.float32(np.float64(vp.softmax_scale(step, step, 64)) * np.log2(np.e))
    S = vt.vitint_qk(slabs[0], slabs[1], batch, heads, tokens)
    P = vt.vitint_softmax_shift_quantize(S.view(batch * heads * tokens, -1), tokens, c2, step_p, bits)
    want = from_codes(vt.vitint_pv(P, slabs[2], batch, heads, tokens, 1.0, 1.0,
                                   vt.Epilogue(mode=vt.EPI_REQUANT, alpha=alpha, out_bits=8, out_signed=True)))
    got = vt.vitint_attention_core_shift(vt.vitint_widen(packed), batch, heads, tokens, step, step, step_p, bits, alpha, None,
                                         out=vt.Codes.empty(batch * tokens, D, 8, True))
    assert np.array_equal(from_codes(got), want)
    from paper_2504_18547_b200.encoder import EncoderLayer
    cfg = si.BlockConfig("steep", 2, tokens, 128, 2, 8, mlp_dim=320)
    layer = EncoderLayer(cfg.batch, tokens, 2, 320, 8, dict(si.layer_parameters(cfg), s_p=step_p))
    x = dev(si.normal(951, (cfg.rows, cfg.dim)))
    out = torch.empty_like(x)
    layer.forward(x, out)
    assert torch.equal(out, one_by_one(layer, x))


@pytest.mark.parametrize("tokens", [33, 197, 256])
@pytest.mark.parametrize("p_step", [1e-3, 1e-4, 2e-5, 1e-5])
def test_shift_core_with_rows_that_peak(tokens, p_step):
    """Keys equal to the queries: one probability near 1, thousands of steps above the last level, beside ones on every level."""
    batch, D, bits, step = 2, 64, 4, np.float32(0.5)
    qkv = rand_codes(970 + tokens, (batch * tokens, 3 * D), bits, True)
    qkv[:, D:2 * D] = qkv[:, :D]
    packed = to_codes(qkv, bits, True)
    slabs = [vt.Slabs.of_qkv(packed, tokens, D, i) for i in range(3)]
    alpha = dev(np.full(D, np.float32(0.02)))
    c2 = np.float32(np.float64(vp.softmax_scale(step, step, 64)) * np.log2(np.e))
    S = vt.vitint_qk(slabs[0], slabs[1], batch, 1, tokens)
    P = vt.vitint_softmax_shift_quantize(S.view(batch * tokens, -1), tokens, c2, np.float32(p_step), bits)
    assert (from_codes(P).max(axis=1) == 15).all()
    want = from_codes(vt.vitint_pv(P, slabs[2], batch, 1, tokens, 1.0, 1.0, vt.Epilogue(mode=vt.EPI_REQUANT, alpha=alpha, out_bits=8, out_signed=True)))
    got = vt.vitint_attention_core_shift(vt.vitint_widen(packed), batch, 1, tokens, step, step, np.float32(p_step), bits, alpha, None,
                                         out=vt.Codes.empty(batch * tokens, D, 8, True))
    assert np.array_equal(from_codes(got), want)


@pytest.mark.parametrize("tokens", [1, 9, 40, 96, 129, 197, 225, 256])
@pytest.mark.parametrize("bits,form", [(4, "byte"), (4, "packed"), (2, "packed"), (4, "shift"), (8, "layer")])
def test_core_with_one_group_and_with_two(tokens, bits, form):
    """Every item with a CTA of its own (one group of sixteen warps) and more items than that (two groups of eight)."""
    heads, D = 2, 128
    batch = torch.cuda.get_device_properties(0).multi_processor_count // (2 * ((tokens + 127) // 128)) + 3
    if form == "layer":
        cfg, layer = small_layer({}, cfg=si.BlockConfig("groups", batch, tokens, D, heads, bits, mlp_dim=320))
        x = dev(si.normal(961, (cfg.rows, cfg.dim)))
        out = torch.empty_like(x)
        layer.forward(x, out)
        assert torch.equal(out, one_by_one(layer, x))
        return
    qkv = to_codes(rand_codes(960 + tokens, (batch * tokens, 3 * D), bits, True), bits, True)
    qkv = qkv if form == "packed" else vt.vitint_widen(qkv)
    alpha, step, p_step = dev(np.full(D, np.float32(0.05))), 0.25, float(np.float32(2.0 / tokens / (2 ** bits - 1) ** 0.5))
    core = vt.vitint_attention_core_shift if form == "shift" else vt.vitint_attention_core
    whole = core(qkv, batch, heads, tokens, step, step, p_step, bits, alpha, None).data
    for first in (0, batch - 3):
        rows = slice(first * tokens, (first + 3) * tokens)
        part = vt.Codes(qkv.data[rows], 3 * tokens, 3 * D, bits, True, qkv.container)
        assert torch.equal(core(part, 3, heads, tokens, step, step, p_step, bits, alpha, None).data, whole[rows])


@pytest.mark.parametrize("tokens,bits", [(1, 4), (15, 2), (16, 4), (24, 4), (32, 2), (40, 3), (197, 4), (256, 3)])
def test_attention_block_qkv_form(tokens, bits):
    """QKV stored one code per byte where its room is that of the unfused sequence, packed otherwise or when a copy is asked for:
    the same output and the same O, twice in a row with the workspace reused (the exp table is filled beside the QKV linear)."""
    cfg = si.BlockConfig("form", 3, tokens, 192, 3, bits)
    prm = si.layer_parameters(cfg)
    xq = vt.vitint_quantize(dev(si.activations(cfg)), float(prm["s_x"]), bits, True)
    w = {n: vt.vitint_quantize(dev(prm["w_" + n]), 0.0, bits, True, row_steps=dev(prm["s_w_" + n])) for n in ("qkv", "proj")}
    seg = np.repeat(np.array([prm["s_q"], prm["s_k"], prm["s_v"]], np.float32), cfg.dim)
    alpha, beta = vt.fold_requant(prm["s_x"], prm["s_w_qkv"], prm["b_qkv"], seg)
    alpha_o, _ = vt.fold_requant(prm["s_p"], np.full(cfg.dim, prm["s_v"], np.float32), None, prm["s_o"])

    def block(step):
        return vt.AttentionWeights(cfg.batch, tokens, cfg.heads, bits, w["qkv"], dev(alpha), dev(beta), step, step, float(prm["s_v"]),
                                   float(prm["s_p"]), float(prm["s_o"]), bits, dev(alpha_o), None, w["proj"], dev(prm["s_w_proj"]),
                                   dev(prm["b_proj"]), vt.Epilogue(mode=vt.EPI_DEQUANT_F32))

    a, b = block(float(prm["s_q"])), block(0.5 * float(prm["s_q"]))
    work = torch.empty(vt.vitint_attention_block_workspace_bytes(a), dtype=torch.uint8, device="cuda")
    want = []
    for d in (a, b):
        copy = vt.Codes.empty(cfg.rows, 3 * cfg.dim, bits, True)
        want.append(vt.vitint_attention_block(xq, d, workspace=work, dbg_qkv=copy))
    got = [vt.vitint_attention_block(xq, d, workspace=work) for _ in range(4) for d in (a, b)]
    assert all(torch.equal(g, want[i % 2]) for i, g in enumerate(got))
    o = [vt.Codes.empty(cfg.rows, cfg.dim, bits, True) for _ in range(2)]
    p = vt.Codes.empty(cfg.batch * cfg.heads * tokens, tokens, bits, False)
    vt.vitint_attention_block(xq, a, workspace=work, dbg_o=o[0])
    vt.vitint_attention_block(xq, a, workspace=work, dbg_o=o[1], dbg_p=p)
    assert torch.equal(o[0].data, o[1].data)


@pytest.mark.parametrize("tokens,q_step", [(40, 1.0), (300, 1.0), (40, 0.1), (300, 0.1)])
def test_attention_block_range_of_the_logits(tokens, q_step):
    """Logits that the exp table cannot hold (the unfused sequence) and logits that it can, with a copy of QKV beside."""
    cfg = si.BlockConfig("range", 2, tokens, 128, 2, 4)
    prm = si.layer_parameters(cfg)
    xq = vt.vitint_quantize(dev(si.activations(cfg)), float(prm["s_x"]), 4, True)
    w = {n: vt.vitint_quantize(dev(prm["w_" + n]), 0.0, 4, True, row_steps=dev(prm["s_w_" + n])) for n in ("qkv", "proj")}
    seg = np.repeat(np.array([prm["s_q"], prm["s_k"], prm["s_v"]], np.float32), cfg.dim)
    alpha, beta = vt.fold_requant(prm["s_x"], prm["s_w_qkv"], prm["b_qkv"], seg)
    alpha_o, _ = vt.fold_requant(prm["s_p"], np.full(cfg.dim, prm["s_v"], np.float32), None, prm["s_o"])
    a = vt.AttentionWeights(cfg.batch, tokens, cfg.heads, 4, w["qkv"], dev(alpha), dev(beta), q_step, q_step, float(prm["s_v"]),
                            float(prm["s_p"]), float(prm["s_o"]), 4, dev(alpha_o), None, w["proj"], dev(prm["s_w_proj"]),
                            dev(prm["b_proj"]), vt.Epilogue(mode=vt.EPI_DEQUANT_F32))
    work = torch.empty(vt.vitint_attention_block_workspace_bytes(a), dtype=torch.uint8, device="cuda")
    p = vt.Codes.empty(cfg.batch * cfg.heads * tokens, tokens, 4, False)
    want = vt.vitint_attention_block(xq, a, dbg_p=p, workspace=work)
    work.fill_(0xA5)
    assert torch.equal(vt.vitint_attention_block(xq, a, workspace=work), want)
    qkv = vt.Codes.empty(cfg.rows, 3 * cfg.dim, 4, True)
    assert torch.equal(vt.vitint_attention_block(xq, a, workspace=work, dbg_qkv=qkv), want)


@pytest.mark.parametrize("rows,cols", [(1, 5), (1183, 768), (1185, 768), (2369, 200), (9473, 33), (4737, 127), (12608, 20), (75781, 12)])
@pytest.mark.parametrize("bits", [2, 3, 4, 8])
def test_quantize_rows_per_thread(rows, cols, bits):
    """Around the row counts from which a thread walks several rows (a remainder of the rows it takes at a time included), values
    on ties, at and beyond the end levels, non-finite."""
    x = si.normal(700 + rows, (rows, cols), 0.0, 3.0)
    step = np.float32(0.25)
    x[::3] = (np.round(x[::3] * 8) / 8).astype(np.float32)                  # ties of the quotient
    flat = x.reshape(-1)
    special = np.array([np.nan, np.inf, -np.inf, 3e38, -3e38, -0.0], np.float32)[:flat.size]
    flat[:special.size] = special
    for signed in (True, False):
        for container in (0, 8):
            out = vt.Codes.empty(rows, cols, bits, signed, container=container)
            out.data.fill_(0x5A)
            vt.vitint_quantize(dev(x), float(step), bits, signed, out=out)
            assert np.array_equal(from_codes(out), vo.quantize(x, step, bits, signed)) and padding_is_zero(out)

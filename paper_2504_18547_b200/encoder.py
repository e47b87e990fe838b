"""Integerized ViT encoder layer as a fixed sequence of C-ABI calls with preallocated buffers.

LayerNorm+quantize -> QKV linear -> Q K^T -> softmax+quantize -> P V -> projection (+residual)
-> LayerNorm+quantize -> fc1 (GELU, requantize) -> fc2 (+residual).  This module only owns
device buffers and marshals arguments; every step runs in the library's kernels.
"""
from __future__ import annotations

import numpy as np
import torch

from . import binding as B

STAGES_UNFUSED = ("ln1_quant", "qkv_linear", "qk", "softmax_quant", "pv", "proj_linear", "ln2_quant", "fc1_linear",
                  "fc2_linear")
STAGES_FUSED = ("ln1_quant", "qkv_linear", "attention_core", "proj_linear", "ln2_quant", "fc1_linear", "fc2_linear")
# stages that run in the integer GEMM kernel
GEMM_STAGES = ("qkv_linear", "qk", "pv", "proj_linear", "fc1_linear", "fc2_linear")


_NO_TENSOR = torch.empty(0)                # stands for an absent tensor where addresses are compared
_data_ptr = torch.Tensor.data_ptr


def _dev(a, device):
    return torch.from_numpy(np.ascontiguousarray(a)).to(device)


class _Recorded:
    """What recorded layers and stacks share: the plan, and the signature of the state it was made for.  Copies and pickles go
    without the plan, which names the original's memory, and make their own at the next forward().  (Class-level values serve
    objects pickled before there were plans.)"""
    _record = False
    _plan = _plan_for = None

    def _planned(self):
        """The plan of the layer or stack as it is now.  None where a stage does not take its shape or steps: forward() then
        launches one by one and reports the error of that stage; it is recorded again once it has changed."""
        if not self._record:
            return None
        now = self._signature()
        if now != self._plan_for:
            if torch.cuda.is_current_stream_capturing():
                return None                # (what making a plan fills would be filled when the captured graph runs)
            self._plan_for, self._plan = now, self._new_plan()
        return self._plan

    def __getstate__(self):
        return {k: v for k, v in self.__dict__.items() if k not in ("_plan", "_plan_for")}


class EncoderLayer(_Recorded):
    _any_core = False
    _sm_table_c = None

    def __init__(self, batch: int, tokens: int, heads: int, mlp_dim: int, bits: int, prm: dict, device="cuda",
                 eps: float = 1e-6, widen_weights: bool = True, fused_attention: bool = True,
                 wide_activations: bool = True, softmax: str = "exp", layernorm: str = "fp32", plan: bool = True):
        """plan: record the layer's launches once as a graph that forward() then launches (a stack records its own)."""
        self.batch, self.tokens, self.heads, self.bits, self.eps = batch, tokens, heads, bits, eps
        self.dim = D = heads * 64
        self.mlp_dim = F = mlp_dim
        self.rows = M = batch * tokens
        self.device = device
        if softmax not in ("exp", "shift"):
            raise ValueError("softmax must be 'exp' (Eq. 3) or 'shift' (Eq. 4 with the comparator quantizer)")
        self.softmax = softmax
        if layernorm not in ("fp32", "compare"):
            raise ValueError("layernorm must be 'fp32' (LayerNorm, then round) or 'compare' (Eq. 5 statistics with the "
                             "division- and square-root-free comparator quantizer)")
        self.layernorm = layernorm
        # the shift-based softmax is a separate kernel: it runs in the unfused attention pipeline
        # the fused core takes the exp softmax for any container and the Eq. 4 softmax for byte-stored codes
        # (beyond 256 tokens the exp core runs its chunked two-pass kernel, which takes byte-stored codes)
        self.fused_attention = (fused_attention and bits != 8
                                and ((softmax == "exp" and (tokens <= 256 or (wide_activations and tokens <= 4096)))
                                     or (softmax == "shift" and wide_activations and tokens <= 256)))
        self.stages = STAGES_FUSED if self.fused_attention else STAGES_UNFUSED
        # 8-bit scores have no table: Q K^T, softmax and P V one by one (as forward() with events times them), or, in the
        # recorded layer, the fused core that evaluates exp per score -- the same codes without S and P in memory, which
        # the layer has only once they are asked for (__getattr__)
        self._any_core = fused_attention and bits == 8 and softmax == "exp" and tokens <= 256
        d = lambda a: _dev(a, device)
        f = lambda k: float(prm[k])
        self.s_ln, self.s_q, self.s_k, self.s_v = f("s_ln"), f("s_q"), f("s_k"), f("s_v")
        self.s_p, self.s_o, self.s_g = f("s_p"), f("s_o"), f("s_g")
        self.ln1_g, self.ln1_b, self.ln2_g, self.ln2_b = d(prm["ln1_g"]), d(prm["ln1_b"]), d(prm["ln2_g"]), d(prm["ln2_b"])
        if layernorm == "compare":
            self.ln_refs = []
            for gk, bk in (("ln1_g", "ln1_b"), ("ln2_g", "ln2_b")):
                r, fl = B.fold_layernorm_references(prm[gk], prm[bk], prm["s_ln"], bits, True, D)
                self.ln_refs.append((d(r), d(fl)))
            self.n_eps = float(np.float32(np.float64(D) * np.float64(np.float32(eps))))
            self.ln_stats = torch.empty((M, 2), dtype=torch.float32, device=device)
        # weights: quantized once by the library's own quantizer (per-output-channel steps)
        self.w = {}
        for name in ("qkv", "proj", "fc1", "fc2"):
            self.w[name] = B.vitint_quantize(d(prm[f"w_{name}"]), 0.0, bits, True, row_steps=d(prm[f"s_w_{name}"]))
        # the low-bit weight codes, re-stored once in 8-bit containers: the GEMM then feeds this
        # operand to the tensor cores straight from the TMA copy
        self.w_packed = dict(self.w)
        if widen_weights and bits != 8:
            self.w = {n: B.vitint_widen(c) for n, c in self.w.items()}
        self.s_w = {n: d(prm[f"s_w_{n}"]) for n in ("proj", "fc1", "fc2")}
        self.bias = {n: d(prm[f"b_{n}"]) for n in ("proj", "fc1", "fc2")}
        seg = np.concatenate([np.full(D, prm["s_q"]), np.full(D, prm["s_k"]), np.full(D, prm["s_v"])]).astype(np.float32)
        a, b = B.fold_requant(prm["s_ln"], prm["s_w_qkv"], prm["b_qkv"], seg)
        self.alpha_qkv, self.beta_qkv = d(a), d(b)
        a, _ = B.fold_requant(prm["s_p"], np.full(D, prm["s_v"], np.float32), None, prm["s_o"])
        self.alpha_o = d(a)
        self.inv_s_g = d((1.0 / np.full(F, prm["s_g"], np.float64)).astype(np.float32))
        self.c = float(np.float32(float(prm["s_q"]) * float(prm["s_k"]) / 8.0))
        self.c2 = float(np.float32(np.float64(np.float32(self.c)) * np.log2(np.e)))   # exponent of two for Eq. 4
        # activations, stored one code per byte: the consumer's TMA copy is then already the
        # tensor-core operand (the unfused attention kernels read packed q, k, v slabs instead)
        ca = 8 if wide_activations and bits != 8 else 0
        cq = ca if self.fused_attention else 0
        self.x1 = B.Codes.empty(M, D, bits, True, device, container=ca)
        self.qkv = B.Codes.empty(M, 3 * D, bits, True, device, container=cq)
        self.ld_s = (tokens + 3) // 4 * 4
        if self.fused_attention and softmax == "shift":
            # (the workspace that the entry point's contract asks for)
            self.attn_table = torch.empty(B.vitint_attention_core_shift_workspace_bytes(bits), dtype=torch.uint8, device=device)
        elif self.fused_attention:
            # the exp table of the fused core depends only on the code width and the steps of Q and K: filled once
            self.attn_table = B.vitint_attention_exp_table(bits, self.s_q, self.s_k, device=device)
        else:
            if not self._any_core:
                self.S, self.P = self._new_scores()
            self._spare_scores = None
            # scores of b-bit codes are bounded by 64 * 2^(b-1) * 2^(b-1): where the table-driven softmax takes that
            # range its exp table is built by the first call and reused afterwards
            half = 1 << ((4 if bits == 3 else bits) - 1)
            self.score_bound = 64 * half * half
            self.sm_table = None
            if (softmax == "exp" and B.vitint_softmax_table_workspace_bytes(self.score_bound) > 0
                    and self.score_bound * abs(self.c) <= 80.0 and tokens <= 895):
                self.sm_table = torch.empty(B.vitint_softmax_table_workspace_bytes(self.score_bound), dtype=torch.uint8,
                                            device=device)
                self.sm_table_ready, self._sm_table_c = False, None
        self.O = B.Codes.empty(M, D, bits, True, device, container=ca)
        self.h = torch.empty((M, D), dtype=torch.float32, device=device)
        self.x2 = B.Codes.empty(M, D, bits, True, device, container=ca)
        self.g = B.Codes.empty(M, F, bits, False, device, container=ca)
        self.slabs = None if self.fused_attention else [B.Slabs.of_qkv(self.qkv, tokens, D, i) for i in range(3)]
        self.epi_qkv = B.Epilogue(mode=B.EPI_REQUANT, alpha=self.alpha_qkv, beta=self.beta_qkv, out_bits=bits,
                                  out_signed=True, out_container=cq)
        self.epi_o = B.Epilogue(mode=B.EPI_REQUANT, alpha=self.alpha_o, out_bits=bits, out_signed=True, out_container=ca)
        self.epi_fc1 = B.Epilogue(mode=B.EPI_REQUANT, act=1, inv_out_step=self.inv_s_g, out_bits=bits, out_signed=False,
                                  out_container=ca)
        self._record = plan
        self._planned()

    def _new_scores(self):
        n = self.batch * self.heads * self.tokens
        return (torch.empty((n, self.ld_s), dtype=torch.int32, device=self.device),
                B.Codes.empty(n, self.tokens, self.bits, False, self.device))

    def _scores(self):
        """S and P for the three attention kernels: the layer's own, or spare ones where forward() does without."""
        if not self._any_core:
            return self.S, self.P
        if self._spare_scores is None:
            self._spare_scores = self._new_scores()
        return self._spare_scores

    def __getattr__(self, name):
        """S and P of an 8-bit layer.  The first time one is asked for, both get the scores and codes of the last call (its QKV
        codes are still there), and from then on forward() keeps them in memory: whoever holds them sees every later call's."""
        if name not in ("S", "P") or not self._any_core:
            raise AttributeError(f"{type(self).__name__!r} object has no attribute {name!r}")
        S, P = self._scores()
        B.vitint_qk(self.slabs[0], self.slabs[1], self.batch, self.heads, self.tokens, out=S, ld_s=self.ld_s)
        B.vitint_softmax_quantize(S, self.tokens, self.c, self.s_p, self.bits, out=P)
        self._any_core, self.S, self.P, self._spare_scores = False, S, P, None
        return self.__dict__[name]

    def _signature(self) -> list:
        """Everything the launches take from this layer, as plain values: the addresses of its weights, parameters and buffers,
        the forms of weights and epilogues, and its scalars.  A plan is used only while it equals the one the plan was made for."""
        w, s, b, eq, eg, none = self.w, self.s_w, self.bias, self.epi_qkv, self.epi_fc1, _NO_TENSOR
        wq, wp, w1, w2 = w["qkv"], w["proj"], w["fc1"], w["fc2"]
        bq, bp, b1, b2 = eq.beta, b["proj"], b["fc1"], b["fc2"]
        t = [self.x1.data, self.qkv.data, self.O.data, self.x2.data, self.g.data, self.h, wq.data, wp.data, w1.data, w2.data,
             s["proj"], s["fc1"], s["fc2"], eq.alpha, eg.inv_out_step, none if bq is None else bq, none if bp is None else bp, none if b1 is None else b1,
             none if b2 is None else b2]
        v = [self.s_ln, self.s_q, self.s_k, self.s_v, self.s_p, self.s_o, self.s_g, self.eps, self.batch, self.tokens,
             wq.container, wp.container, w1.container, w2.container, eq.mode, eq.act, eq.out_bits, eq.out_signed, eq.out_container,
             eg.mode, eg.act, eg.out_bits, eg.out_signed, eg.out_container]
        if self.layernorm == "compare":
            (r1, f1), (r2, f2) = self.ln_refs
            t += [r1, r2, self.ln_stats, none if f1 is None else f1, none if f2 is None else f2]
            v.append(self.n_eps)
        else:
            t += [self.ln1_g, self.ln1_b, self.ln2_g, self.ln2_b]
        if self.fused_attention:
            t += [self.alpha_o, self.attn_table]
        else:
            eo = self.epi_o
            t += [eo.alpha, none if eo.beta is None else eo.beta]
            v += [eo.mode, eo.act, eo.out_bits, eo.out_signed, eo.out_container, self.c, self.c2, self._any_core]
            if not self._any_core:
                t += [self.S, self.P.data]
                v += [self.P.container, self.ld_s, self.score_bound]
                if self.sm_table is not None:
                    t.append(self.sm_table)
        v.extend(map(_data_ptr, t))
        return v

    def _recordable(self) -> bool:
        """Whether the epilogues are of the form that a recorded layer gives them (forward() takes any)."""
        def form(e, codes, act, signed):
            return (e.mode, e.act, e.out_bits, bool(e.out_signed), e.out_container) == (B.EPI_REQUANT, act, codes.bits, signed, codes.container)
        return (form(self.epi_qkv, self.qkv, 0, True) and form(self.epi_fc1, self.g, 1, False)
                and (self.fused_attention or (form(self.epi_o, self.O, 0, True) and self.epi_o.beta is None)))

    def _desc(self):
        d = B._EncoderLayerDesc()
        d.batch, d.tokens, d.heads, d.bits = self.batch, self.tokens, self.heads, self.bits
        d.eps, d.ln_step, d.g_step = self.eps, self.s_ln, self.s_g
        d.q_step, d.k_step, d.v_step, d.p_step, d.o_step = self.s_q, self.s_k, self.s_v, self.s_p, self.s_o
        p = B._ptr
        if self.layernorm == "compare":
            d.compare_layernorm, d.n_eps, d.ln_stats = 1, self.n_eps, p(self.ln_stats)
            (r1, f1), (r2, f2) = self.ln_refs
            d.ln1_refs, d.ln1_flip, d.ln2_refs, d.ln2_flip = p(r1), p(f1), p(r2), p(f2)
        else:
            d.ln1_gamma, d.ln1_beta, d.ln2_gamma, d.ln2_beta = p(self.ln1_g), p(self.ln1_b), p(self.ln2_g), p(self.ln2_b)
        d.w_qkv, d.w_proj, d.w_fc1, d.w_fc2 = (self.w[n].desc() for n in ("qkv", "proj", "fc1", "fc2"))
        d.alpha_qkv, d.beta_qkv, d.inv_g_step = p(self.epi_qkv.alpha), p(self.epi_qkv.beta), p(self.epi_fc1.inv_out_step)
        d.alpha_o = p(self.alpha_o if self.fused_attention else self.epi_o.alpha)
        d.proj_step, d.fc1_step, d.fc2_step = (p(self.s_w[n]) for n in ("proj", "fc1", "fc2"))
        d.proj_bias, d.fc1_bias, d.fc2_bias = (p(self.bias[n]) for n in ("proj", "fc1", "fc2"))
        d.x1, d.qkv, d.o, d.x2, d.g = self.x1.desc(), self.qkv.desc(), self.O.desc(), self.x2.desc(), self.g.desc()
        d.h = p(self.h)
        table = None
        if self.fused_attention:
            d.attention = B.ATTN_SHIFT_CORE if self.softmax == "shift" else B.ATTN_EXP_CORE
            table = self.attn_table
        elif self._any_core:
            d.attention = B.ATTN_EXP_CORE_ANY
        else:
            d.scores, d.ld_scores, d.p = p(self.S), self.ld_s, self.P.desc()
            if self.softmax == "shift":
                d.attention, d.c = B.ATTN_SHIFT, self.c2
            elif self.sm_table is not None:
                d.attention, d.c, d.score_bound, table = B.ATTN_EXP_BOUNDED, self.c, self.score_bound, self.sm_table
            else:
                d.attention, d.c = B.ATTN_EXP, self.c
        if table is not None:
            d.table, d.table_bytes = p(table), table.numel()
        return d

    def _tables_filled(self):
        """Making a plan fills the tables of the attention variants that build theirs on first use."""
        if not self.fused_attention and self.sm_table is not None:
            self.sm_table_ready, self._sm_table_c = True, self.c

    def _new_plan(self):
        if not self._recordable():
            return None
        try:
            plan = B.EncoderPlan([self._desc()])
        except B.VitintError:
            return None
        self._tables_filled()
        return plan

    def _plain_io(self, x: torch.Tensor, out: torch.Tensor) -> bool:
        """Whether x and out are dense matrices of the layer's shape (what a plan takes)."""
        shape = (self.rows, self.dim)
        return x.shape == shape and out.shape == shape and x.is_contiguous() and out.is_contiguous()

    def forward(self, x: torch.Tensor, out: torch.Tensor, events: list | None = None) -> torch.Tensor:
        """x, out: fp32 [batch*tokens, dim] on the device.  `events`, when given, receives
        len(self.stages)+1 recorded CUDA events bracketing the stages (of an 8-bit layer too: Q K^T, softmax and P V, where
        a call without events runs one kernel with the same codes)."""
        plan = self._planned() if events is None and self._plain_io(x, out) else None
        if plan is not None:
            plan.run(x, out)
            return out
        def mark():
            if events is not None:
                e = torch.cuda.Event(enable_timing=True)
                e.record()
                events.append(e)
        b, t, h = self.batch, self.tokens, self.heads
        mark()
        if self.layernorm == "compare":
            B.vitint_layernorm_compare_quantize(x, self.ln_refs[0][0], self.ln_refs[0][1], self.n_eps, self.bits, True,
                                                out=self.x1, stats=self.ln_stats)
        else:
            B.vitint_layernorm_quantize(x, self.ln1_g, self.ln1_b, self.eps, self.s_ln, self.bits, True, out=self.x1)
        mark()
        B.vitint_linear(self.x1, self.s_ln, self.w["qkv"], None, None, self.epi_qkv, out=self.qkv)
        mark()
        if self.fused_attention and self.softmax == "shift":
            B.vitint_attention_core_shift(self.qkv, b, h, t, self.s_q, self.s_k, self.s_p, self.bits, self.alpha_o, None,
                                          out=self.O, workspace=self.attn_table)
        elif self.fused_attention:
            B.vitint_attention_core_prepared(self.qkv, b, h, t, self.s_q, self.s_k, self.s_p, self.bits, self.alpha_o,
                                             None, out=self.O, table=self.attn_table)
        else:
            S, P = self._scores()
            B.vitint_qk(self.slabs[0], self.slabs[1], b, h, t, out=S, ld_s=self.ld_s)
            mark()
            if self.softmax == "shift":
                B.vitint_softmax_shift_quantize(S, t, self.c2, self.s_p, self.bits, out=P)
            elif self.sm_table is not None:
                ready = self.sm_table_ready and self._sm_table_c == self.c
                B.vitint_softmax_quantize_bounded(S, t, self.c, self.s_p, self.bits, self.score_bound, out=P,
                                                  workspace=self.sm_table, table_ready=ready)
                if not ready and not torch.cuda.is_current_stream_capturing():     # (a captured launch fills it when its graph runs)
                    self._tables_filled()
            else:
                B.vitint_softmax_quantize(S, t, self.c, self.s_p, self.bits, out=P)
            mark()
            B.vitint_pv(P, self.slabs[2], b, h, t, self.s_p, self.s_v, self.epi_o, out=self.O)
        mark()
        B.vitint_linear(self.O, self.s_o, self.w["proj"], self.s_w["proj"], self.bias["proj"],
                        B.Epilogue(mode=B.EPI_DEQUANT_F32, residual=x), out=self.h)
        mark()
        if self.layernorm == "compare":
            B.vitint_layernorm_compare_quantize(self.h, self.ln_refs[1][0], self.ln_refs[1][1], self.n_eps, self.bits,
                                                True, out=self.x2, stats=self.ln_stats)
        else:
            B.vitint_layernorm_quantize(self.h, self.ln2_g, self.ln2_b, self.eps, self.s_ln, self.bits, True, out=self.x2)
        mark()
        B.vitint_linear(self.x2, self.s_ln, self.w["fc1"], self.s_w["fc1"], self.bias["fc1"], self.epi_fc1, out=self.g)
        mark()
        B.vitint_linear(self.g, self.s_g, self.w["fc2"], self.s_w["fc2"], self.bias["fc2"],
                        B.Epilogue(mode=B.EPI_DEQUANT_F32, residual=self.h), out=out)
        mark()
        return out

    def stage_ops(self) -> dict:
        """Integer operations (2 per multiply-accumulate, true shapes) of each contraction."""
        M, D, F, T = self.rows, self.dim, self.mlp_dim, self.tokens
        n = self.batch * self.heads
        return {"qkv_linear": 2 * M * D * 3 * D, "qk": 2 * n * T * T * 64, "pv": 2 * n * T * T * 64,
                "attention_core": 4 * n * T * T * 64, "proj_linear": 2 * M * D * D, "fc1_linear": 2 * M * D * F,
                "fc2_linear": 2 * M * F * D}

    def stage_bytes(self) -> dict:
        """Algorithmic HBM bytes of the streaming stages (4 + c/8 per element)."""
        c = 4 if self.bits == 3 else self.bits
        cx = self.x1.stored_bits
        M, D, T = self.rows, self.dim, self.tokens
        n = self.batch * self.heads * T
        return {"ln1_quant": M * D * 4 + M * D * cx // 8, "ln2_quant": M * D * 4 + M * D * cx // 8,
                "softmax_quant": n * T * 4 + n * ((T * c + 7) // 8)}


class EncoderStack(_Recorded):
    """`layers` integerized encoder layers applied in sequence (each with its own weights and steps);
    the fp32 residual stream ping-pongs between two device buffers."""

    def __init__(self, layer_params: list, batch: int, tokens: int, heads: int, mlp_dim: int, bits: int,
                 device="cuda", **kw):
        plan, kw = kw.get("plan", True), dict(kw, plan=False)       # (recorded as a whole)
        self.layers = [EncoderLayer(batch, tokens, heads, mlp_dim, bits, prm, device, **kw) for prm in layer_params]
        rows, dim = batch * tokens, heads * 64
        self.buf = [torch.empty((rows, dim), dtype=torch.float32, device=device) for _ in range(2)]
        self._record = plan and bool(self.layers)
        self._planned()

    def _signature(self) -> list:
        return [l._signature() for l in self.layers] + [b.data_ptr() for b in self.buf]

    def _new_plan(self):
        if not all(l._recordable() for l in self.layers):
            return None
        try:
            plan = B.EncoderPlan([l._desc() for l in self.layers], self.buf)
        except B.VitintError:
            return None
        for l in self.layers:
            l._tables_filled()
        return plan

    def forward(self, x: torch.Tensor, out: torch.Tensor) -> torch.Tensor:
        plan = self._planned() if self._record and self.layers[0]._plain_io(x, out) else None
        if plan is not None:
            plan.run(x, out)
            return out
        cur = x
        n = len(self.layers)
        for i, layer in enumerate(self.layers):
            dst = out if i == n - 1 else self.buf[i & 1]
            layer.forward(cur, dst)
            cur = dst
        return out

    def ops(self) -> int:
        return sum(sum(v for k, v in l.stage_ops().items() if k in l.stages) for l in self.layers)


class NormedAttention:
    """The self-attention module laid out as in the paper's power table (Section V-B): separate Q, K and V
    linear layers, a LayerNorm over each head's 64 channels in front of the Q and K quantizers (statistics by
    Eq. 5, comparator quantizer of Fig. 5(b)), Q K^T, the Eq. 4 softmax with its division-free quantizer, P V.
    A fixed sequence of C-ABI calls over preallocated buffers; `qkn` holds the per-head LayerNorm parameters
    (qn_g, qn_b, kn_g, kn_b over 64 channels) and the steps s_qn, s_kn of the normalised values.
    fused=True (default): one QKV GEMM whose epilogue normalises and quantizes the Q and K heads and requantizes V,
    then the fused attention core with the Eq. 4 softmax inside (2 launches; `fused_core=False` keeps Q K^T, softmax
    and P V as three kernels with S and P in memory: 4 launches); fused=False: separate Q, K, V linears with fp32 Q
    and K rows and a LayerNorm kernel each (8 launches, the fp32 rows and their statistics left in `f32` /
    `stats` for inspection)."""

    def __init__(self, batch: int, tokens: int, heads: int, bits: int, prm: dict, qkn: dict, device="cuda",
                 eps: float = 1e-6, fused: bool = True, fused_core: bool = True):
        self.fused = fused
        self.fused_core = fused and fused_core and tokens <= 256 and bits != 8
        self.batch, self.tokens, self.heads, self.bits = batch, tokens, heads, bits
        self.dim = D = heads * 64
        self.rows = M = batch * tokens
        d = lambda a: _dev(a, device)
        w = B.vitint_widen(B.vitint_quantize(d(prm["w_qkv"]), 0.0, bits, True, row_steps=d(prm["s_w_qkv"])))
        part = lambda i: B.Codes(w.data[i * D:(i + 1) * D], D, D, bits, True, 8)
        self.w_qkv, self.w_q, self.w_k, self.w_v = w, part(0), part(1), part(2)
        self.s_w_all, self.bias_all = d(prm["s_w_qkv"]), d(prm["b_qkv"])
        self.s_w = [self.s_w_all[i * D:(i + 1) * D] for i in range(2)]
        self.bias = [self.bias_all[i * D:(i + 1) * D] for i in range(2)]
        a, b = B.fold_requant(1.0, prm["s_w_qkv"][2 * D:], prm["b_qkv"][2 * D:], prm["s_v"])
        self._alpha_v_unit, self.beta_v = a, d(b)             # alpha scales with the input step given to forward()
        self.refs = []
        for n in ("q", "k"):
            r, fl = B.fold_layernorm_references(qkn[n + "n_g"], qkn[n + "n_b"], qkn["s_" + n + "n"], bits, True, 64)
            self.refs.append((d(r), d(fl)))
        self.refs_all = torch.stack([r for r, _ in self.refs]).contiguous()
        self.flip_all = torch.stack([f for _, f in self.refs]).contiguous()
        self.n_eps = float(np.float32(np.float64(64) * np.float64(np.float32(eps))))
        self.s_v, self.s_p, self.s_o = float(prm["s_v"]), float(prm["s_p"]), float(prm["s_o"])
        c = np.float32(float(qkn["s_qn"]) * float(qkn["s_kn"]) / 8.0)
        self.c2 = float(np.float32(np.float64(c) * np.log2(np.e)))
        a_o, _ = B.fold_requant(prm["s_p"], np.full(D, prm["s_v"], np.float32), None, prm["s_o"])
        self.alpha_o = d(a_o)
        self._prm = prm
        self._alpha_v_for = None
        c_bits = 4 if bits == 3 else bits
        self.stats_all = torch.empty((2, M * heads, 2), dtype=torch.float32, device=device)
        self.stats = [self.stats_all[0], self.stats_all[1]]
        pitch = D * c_bits // 8
        if self.fused_core:
            # byte-stored QKV codes: the operand form of the fused core
            self.qkv = B.Codes.empty(M, 3 * D, bits, True, device, container=8)
            self.core_ws = torch.empty(B.vitint_attention_core_shift_workspace_bytes(bits), dtype=torch.uint8, device=device)
            self.slabs = self.v_slabs = None
        elif fused:
            self.qkv = B.Codes.empty(M, 3 * D, bits, True, device)
            qp = self.qkv.pitch
            self.slabs = [B.Slabs(self.qkv.data, i * pitch, qp, qp * tokens, 64 * c_bits // 8, bits, True) for i in range(2)]
            self.v_slabs = B.Slabs(self.qkv.data, 2 * pitch, qp, qp * tokens, 64 * c_bits // 8, bits, True)
        else:
            self.f32 = [torch.empty((M, D), dtype=torch.float32, device=device) for _ in range(2)]
            self.qk_codes = [B.Codes.empty(M * heads, 64, bits, True, device) for _ in range(2)]
            self.slabs = [B.Slabs(c.data, 0, pitch, pitch * tokens, 64 * c_bits // 8, bits, True) for c in self.qk_codes]
            self.v = B.Codes.empty(M, D, bits, True, device)
            self.v_slabs = B.Slabs(self.v.data, 0, self.v.pitch, self.v.pitch * tokens, 64 * c_bits // 8, bits, True)
        self.ld_s = (tokens + 3) // 4 * 4
        if not self.fused_core:
            self.S = torch.empty((batch * heads * tokens, self.ld_s), dtype=torch.int32, device=device)
            self.P = B.Codes.empty(batch * heads * tokens, tokens, bits, False, device)
        self.O = B.Codes.empty(M, D, bits, True, device)
        self.epi_o = B.Epilogue(mode=B.EPI_REQUANT, alpha=self.alpha_o, out_bits=bits, out_signed=True)
        self.s_qn, self.s_kn = float(qkn["s_qn"]), float(qkn["s_kn"])

    def forward(self, x: "B.Codes", s_x: float) -> "B.Codes":
        """x: codes [batch*tokens, dim] with step s_x.  Returns the O codes [batch*tokens, dim]."""
        if self._alpha_v_for != float(s_x):
            D = self.dim
            a, _ = B.fold_requant(s_x, self._prm["s_w_qkv"][2 * D:], None, self._prm["s_v"])
            self.alpha_v = _dev(a, self.O.data.device)
            self._alpha_v_for = float(s_x)
        b, t, h = self.batch, self.tokens, self.heads
        if self.fused:
            B.vitint_linear_qkv_norm(x, s_x, self.w_qkv, self.s_w_all, self.bias_all, self.refs_all, self.flip_all,
                                     self.n_eps, self.alpha_v, self.beta_v, self.bits, out=self.qkv, stats=self.stats_all)
        else:
            for i, w in enumerate((self.w_q, self.w_k)):
                B.vitint_linear(x, s_x, w, self.s_w[i], self.bias[i], B.Epilogue(mode=B.EPI_DEQUANT_F32), out=self.f32[i])
                B.vitint_layernorm_compare_quantize(self.f32[i].view(self.rows * h, 64), self.refs[i][0], self.refs[i][1],
                                                    self.n_eps, self.bits, True, out=self.qk_codes[i], stats=self.stats[i])
            B.vitint_linear(x, s_x, self.w_v, None, None,
                            B.Epilogue(mode=B.EPI_REQUANT, alpha=self.alpha_v, beta=self.beta_v, out_bits=self.bits,
                                       out_signed=True), out=self.v)
        if self.fused_core:
            B.vitint_attention_core_shift(self.qkv, b, h, t, self.s_qn, self.s_kn, self.s_p, self.bits, self.alpha_o, None,
                                          out=self.O, workspace=self.core_ws)
            return self.O
        B.vitint_qk(self.slabs[0], self.slabs[1], b, h, t, out=self.S, ld_s=self.ld_s)
        B.vitint_softmax_shift_quantize(self.S, t, self.c2, self.s_p, self.bits, out=self.P)
        B.vitint_pv(self.P, self.v_slabs, b, h, t, self.s_p, self.s_v, self.epi_o, out=self.O)
        return self.O

    def ops(self) -> int:
        """Integer operations (2 per multiply-accumulate) of the five contractions."""
        M, D, T = self.rows, self.dim, self.tokens
        return 2 * (3 * M * D * D + 2 * self.batch * self.heads * T * T * 64)


class DeitModel:
    """The whole DeiT-S-shaped model as C-ABI calls: quantize the flattened patches, patch embedding as an
    integerized linear whose fp32 epilogue adds the token table (class / distillation tokens and position
    embeddings; the two token rows of every image carry zero patches), the encoder layers, final LayerNorm +
    quantizer on the class and distillation rows, two classifier heads (the second adds onto the first's logits)."""

    def __init__(self, ends: dict, layer_params: list, batch: int, tokens: int, heads: int, mlp_dim: int, bits: int,
                 device="cuda", eps: float = 1e-6, **layer_kw):
        self.batch, self.tokens, self.bits, self.eps = batch, tokens, bits, eps
        self.dim = D = heads * 64
        M = batch * tokens
        d = lambda a: _dev(a, device)
        self.stack = EncoderStack(layer_params, batch, tokens, heads, mlp_dim, bits, device, eps=eps, **layer_kw)
        q = lambda w, s: B.vitint_widen(B.vitint_quantize(d(w), 0.0, bits, True, row_steps=d(s)))
        self.w_pe, self.s_w_pe, self.b_pe = q(ends["w_pe"], ends["s_w_pe"]), d(ends["s_w_pe"]), d(ends["b_pe"])
        self.table = d(np.tile(np.asarray(ends["tokens"], np.float32), (batch, 1)))
        self.s_patch, self.s_lnf = float(ends["s_patch"]), float(ends["s_lnf"])
        self.lnf_g, self.lnf_b = d(ends["lnf_g"]), d(ends["lnf_b"])
        self.heads_w = [(q(ends["w_" + n], ends["s_w_" + n]), d(ends["s_w_" + n]), d(ends["b_" + n]))
                        for n in ("head", "head_dist")]
        n_cls = ends["w_head"].shape[0]
        self.xq = B.Codes.empty(M, ends["w_pe"].shape[1], bits, True, device, container=8)
        self.x0 = torch.empty((M, D), dtype=torch.float32, device=device)
        self.x_final = torch.empty((M, D), dtype=torch.float32, device=device)
        self.head_codes = [B.Codes.empty(batch, D, bits, True, device, container=8) for _ in range(2)]
        self.logits = [torch.empty((batch, n_cls), dtype=torch.float32, device=device) for _ in range(2)]

    def forward(self, patches: torch.Tensor) -> torch.Tensor:
        """patches: fp32 [batch*tokens, patch_dim] on the device.  Returns the summed logits [batch, classes]."""
        B.vitint_quantize(patches, self.s_patch, self.bits, True, out=self.xq)
        B.vitint_linear(self.xq, self.s_patch, self.w_pe, self.s_w_pe, self.b_pe,
                        B.Epilogue(mode=B.EPI_DEQUANT_F32, residual=self.table), out=self.x0)
        self.stack.forward(self.x0, self.x_final)
        for i, (w, s_w, b) in enumerate(self.heads_w):
            rows = self.x_final[i::self.tokens]                 # class rows (i = 0), distillation rows (i = 1)
            B.vitint_layernorm_quantize(rows, self.lnf_g, self.lnf_b, self.eps, self.s_lnf, self.bits, True,
                                        out=self.head_codes[i])
            B.vitint_linear(self.head_codes[i], self.s_lnf, w, s_w, b,
                            B.Epilogue(mode=B.EPI_DEQUANT_F32, residual=self.logits[0] if i else None),
                            out=self.logits[i])
        return self.logits[1]

    def ops(self) -> int:
        M, D = self.batch * self.tokens, self.dim
        ends = 2 * M * D * self.xq.cols + 2 * 2 * self.batch * D * self.logits[0].shape[1]
        return ends + self.stack.ops()

"""The warm-start U-Net: a 4-level BF16 network trained and run by the library's own
tensor-core kernels (include/tpfnet.h).  This module only allocates buffers (torch
tensors), orders the kernel calls and marshals arguments; every layer, gradient and
optimizer update runs in CUDA.

Network (channels c0..c3, NHWC bf16, input channels padded to 32):
  e0 = relu(conv(relu(conv(x))))            e1 = ... (pool(e0))     e2 = ... (pool(e1))
  b  = relu(conv(relu(conv(pool(e2)))))
  d2 = relu(conv(relu(conv(cat(up(b), e2)))))   d1 = ... cat(up(d2), e1)   d0 = ... cat(up(d1), e0)
  out = head(d0)  (1x1, float32)
"""
from __future__ import annotations

import ctypes as C

import numpy as np

from .tpflbm import load_library

_vp, _ip, _ll, _fl = C.c_void_p, C.c_int, C.c_longlong, C.c_float
_fp, _dp = C.POINTER(C.c_float), C.POINTER(C.c_double)

SIGNATURES = {
    "tpfnet_conv3x3": [_vp, _ip, _ip, _ip, _ip, _vp, _vp, _ip, _ip, _vp, _vp],
    "tpfnet_conv3x3_into": [_vp, _ip, _ip, _ip, _ip, _vp, _vp, _ip, _ip, _vp, _ip, _vp],
    "tpfnet_conv3x3_dgrad_masked": [_vp, _ip, _ip, _ip, _ip, _vp, _ip, _vp, _vp, _vp],
    "tpfnet_flip_weights": [_ip, _vp, _vp, _vp, _vp, _vp],
    "tpfnet_pool_from": [_vp, _ip, _ip, _ip, _ip, _ip, _vp, _vp],
    "tpfnet_pool_back_skip": [_vp, _ip, _ip, _ip, _ip, _vp, _ip, _vp, _ip, _vp, _vp],
    "tpfnet_up_back_masked": [_vp, _ip, _ip, _ip, _ip, _ip, _ip, _vp, _vp, _vp],
    "tpfnet_head_back_masked": [_vp, _vp, _ll, _ip, _vp, _ip, _vp, _vp, _vp, _vp],
    "tpfnet_unet_forward": [_vp, _vp, _ip, _ip, _ip, _vp, _vp],
    "tpfnet_wgrad_parts": [_ip, _ip, _ip, _ip, _ip],
    "tpfnet_conv3x3_wgrad_part": [_vp, _vp, _ip, _ip, _ip, _ip, _ip, _vp, _vp],
    "tpfnet_head_parts": [_ll, _ip, _ip],
    "tpfnet_head_back_part": [_vp, _vp, _ll, _ip, _vp, _ip, _vp, _vp, _vp],
    "tpfnet_sum_parts": [_ip, _vp, _vp, _vp, _vp, _vp, _vp],
    "tpfnet_conv3x3_tcgen05": [_ip, _ip, _ip, _ip, _ip],
    "tpfnet_conv3x3_wgrad_tcgen05": [_ip, _ip, _ip, _ip, _ip],
    "tpfnet_status": [],
    "tpfnet_check_bounded_wait": [_ip, _vp],
    "tpfnet_conv3x3_dgrad": [_vp, _ip, _ip, _ip, _ip, _vp, _ip, _vp, _vp, _vp],
    "tpfnet_conv3x3_wgrad": [_vp, _vp, _ip, _ip, _ip, _ip, _ip, _vp, _vp, _vp],
    "tpfnet_relu_mask": [_vp, _vp, _ll, _vp],
    "tpfnet_pool": [_vp, _ip, _ip, _ip, _ip, _vp, _vp],
    "tpfnet_pool_back": [_vp, _ip, _ip, _ip, _ip, _vp, _ip, _vp],
    "tpfnet_up_into": [_vp, _ip, _ip, _ip, _ip, _vp, _ip, _ip, _vp],
    "tpfnet_up_back": [_vp, _ip, _ip, _ip, _ip, _ip, _ip, _vp, _vp],
    "tpfnet_channels": [_vp, _ip, _ip, _ll, _ip, _vp, _ip, _ip, _ip, _vp],
    "tpfnet_head": [_vp, _ll, _ip, _vp, _vp, _ip, _vp, _vp],
    "tpfnet_head_back": [_vp, _vp, _ll, _ip, _vp, _ip, _vp, _vp, _vp, _vp],
    "tpfnet_mse": [_vp, _vp, _vp, _ll, _ip, _vp, _vp, _vp],
    "tpfnet_adam": [_vp, _vp, _vp, _vp, _ll, _fl, _fl, _fl, _fl, _ip, _vp, _vp],
    "tpfnet_to_bf16": [_vp, _ll, _vp, _vp],
    "tpfnet_pack": [_vp, _vp, _ll, _ip, _ll, _vp, _vp, _vp, _ip, _ip, _vp],
    "tpfnet_unpack": [_vp, _ll, _ip, _vp, _vp, _vp, _vp, _ll, _vp],
}


class _Net(C.Structure):
    """tpfnet_unet"""
    _fields_ = [("cin", _ip), ("cout", _ip), ("ch", _ip * 4), ("weight", _vp * 14), ("bias", _vp * 14),
                ("head_w", _vp), ("head_b", _vp), ("enc", _vp * 4), ("pool", _vp * 3), ("cat", _vp * 3),
                ("deep", _vp), ("dec_a", _vp * 3), ("dec", _vp * 3)]


PAD = 32  # channel granularity of the convolution kernels


def net_library():
    lib = load_library()
    for name, args in SIGNATURES.items():
        fn = getattr(lib, name)
        fn.argtypes = args
        fn.restype = C.c_int
    return lib


def _p(t):
    return None if t is None else C.c_void_p(t.data_ptr())


def layer_specs(cin, cout, ch):
    """(name, Cin, Cout, taps) of every layer; Cin padded to the kernel granularity."""
    c0, c1, c2, c3 = ch
    cinp = -(-cin // PAD) * PAD
    spec = [("e0a", cinp, c0), ("e0b", c0, c0), ("e1a", c0, c1), ("e1b", c1, c1),
            ("e2a", c1, c2), ("e2b", c2, c2), ("b_a", c2, c3), ("b_b", c3, c3),
            ("d2a", c3 + c2, c2), ("d2b", c2, c2), ("d1a", c2 + c1, c1), ("d1b", c1, c1),
            ("d0a", c1 + c0, c0), ("d0b", c0, c0)]
    return [(n, a, b, 9) for n, a, b in spec] + [("head", c0, cout, 1)]


class UNet:
    def __init__(self, cin, cout, ch=(32, 64, 128, 256), seed=0, stream=None):
        import torch

        if not torch.cuda.is_available():
            raise RuntimeError("the U-Net kernels need a CUDA device")
        for c in ch:
            assert c % 64 == 0 or c == 32, "level channels: 32 or multiples of 64"
        self.torch = torch
        self.lib = net_library()
        self.cin, self.cout, self.ch = cin, cout, tuple(ch)
        self.cinp = -(-cin // PAD) * PAD
        self.specs = layer_specs(cin, cout, ch)
        self.stream = stream if stream is not None else torch.cuda.current_stream()
        rng = np.random.default_rng(seed)
        self.P, self.Pb, self.G, self.M, self.V = {}, {}, {}, {}, {}
        # every parameter is a view into one flat tensor per kind (each starting on a 256-byte
        # boundary), so that Adam and clearing the gradients are one launch each
        total = sum(-(-taps * a * b // 128) * 128 + -(-b // 128) * 128 for _, a, b, taps in self.specs)
        self._flat = {k: torch.zeros(total, dtype=torch.bfloat16 if k == "Pb" else torch.float32, device="cuda")
                      for k in ("P", "G", "M", "V", "Pb")}
        self._used = 0
        for name, a, b, taps in self.specs:
            fan_in = taps * (self.cin if name == "e0a" else a)
            w = rng.standard_normal((taps, b, a) if taps == 9 else (a, b)) * np.sqrt(2.0 / fan_in)
            if name == "e0a":
                w[:, :, cin:] = 0.0
            self._add(name + ".W", w.astype(np.float32), bf16=(taps == 9))
            self._add(name + ".b", (0.01 * rng.standard_normal(b)).astype(np.float32), bf16=False)
        self.adam_t = 0
        self._shape = None
        # all of that was queued on the current stream
        self.stream.wait_stream(torch.cuda.current_stream())

    def _on_stream(self):
        """torch's current stream is the network's own inside: what torch clears, copies and
        reads between the kernels is ordered with them."""
        return self.torch.cuda.stream(self.stream)

    def _add(self, key, arr, bf16):
        t = self.torch
        n, o = arr.size, self._used
        self._used += -(-n // 128) * 128
        for kind in ("P", "G", "M", "V", "Pb"):
            getattr(self, kind)[key] = self._flat[kind][o:o + n].view(arr.shape)
        self.P[key].copy_(t.from_numpy(np.ascontiguousarray(arr)))
        self.Pb[key].copy_(self.P[key])
        if not bf16:
            self.Pb[key] = None

    def _is_flat(self, kinds):
        """Whether every tensor of these kinds is still the view into its flat tensor that
        _add made (a caller may have put tensors of its own in their place)."""
        o = 0
        for name, a, b, taps in self.specs:
            for key, n in ((name + ".W", taps * a * b), (name + ".b", b)):
                for kind in kinds:
                    v, f = getattr(self, kind)[key], self._flat[kind]
                    if v is not None and (v.numel() != n or v.data_ptr() != f.data_ptr() + o * f.element_size()):
                        return False
                o += -(-n // 128) * 128
        return True

    # ------------------------------------------------------- parameter I/O
    def set_reference_params(self, params):
        """Load parameters in the numpy reference layout (W[dh][dw][ci][co])."""
        for name, a, b, taps in self.specs:
            W = params[name + ".W"]
            if taps == 9:
                w = np.zeros((9, b, a), dtype=np.float32)
                w[:, :, :W.shape[2]] = W.reshape(9, W.shape[2], b).transpose(0, 2, 1)
            else:
                w = W.reshape(W.shape[2], b).astype(np.float32)
            self.P[name + ".W"].copy_(self.torch.from_numpy(w))
            if taps == 9:
                self.Pb[name + ".W"].copy_(self.P[name + ".W"].to(self.torch.bfloat16))
            self.P[name + ".b"].copy_(self.torch.from_numpy(params[name + ".b"].astype(np.float32)))

    def reference_grads(self):
        """Gradients in the numpy reference layout."""
        out = {}
        for name, a, b, taps in self.specs:
            g = self.G[name + ".W"].cpu().numpy().astype(np.float64)
            if taps == 9:
                ci = self.cin if name == "e0a" else a
                out[name + ".W"] = g.transpose(0, 2, 1)[:, :ci, :].reshape(3, 3, ci, b)
            else:
                out[name + ".W"] = g.reshape(1, 1, a, b)
            out[name + ".b"] = self.G[name + ".b"].cpu().numpy().astype(np.float64)
        return out

    def state_dict(self):
        return {k: v.cpu().numpy() for k, v in self.P.items()}

    def load_state_dict(self, d):
        for k, v in d.items():
            self.P[k].copy_(self.torch.from_numpy(v))
            if self.Pb[k] is not None:
                self.Pb[k].copy_(self.P[k].to(self.torch.bfloat16))

    # ---------------------------------------------------------- buffers
    def _buffers(self, N, H, W):
        if self._shape == (N, H, W):
            return
        assert H % 8 == 0 and W % 64 == 0, "H multiple of 8, W multiple of 64"
        with self._on_stream():
            self._new_buffers(N, H, W)

    def _new_buffers(self, N, H, W):
        t = self.torch
        c0, c1, c2, c3 = self.ch
        bf = dict(dtype=t.bfloat16, device="cuda")
        self.B = {}
        dims = [(H, W, c0), (H // 2, W // 2, c1), (H // 4, W // 4, c2), (H // 8, W // 8, c3)]
        for lvl, (h, w, c) in enumerate(dims):
            nm = ["e0", "e1", "e2", "b"][lvl]
            self.B[nm + "a"] = t.empty((N, h, w, c), **bf)
            if lvl == 3:
                self.B[nm] = t.empty((N, h, w, c), **bf)
            if lvl > 0:
                cin = dims[lvl - 1][2]
                self.B["pool%d" % lvl] = t.empty((N, h, w, cin), **bf)
        for lvl, (h, w, c) in ((2, dims[2]), (1, dims[1]), (0, dims[0])):
            cup = dims[lvl + 1][2] if lvl == 2 else self.ch[lvl + 1]
            self.B["cat%d" % lvl] = t.empty((N, h, w, cup + c), **bf)
            # the encoder's output is the concatenation's second part (written there)
            self.B["e%d" % lvl] = self.B["cat%d" % lvl][..., cup:]
            self.B["d%da" % lvl] = t.empty((N, h, w, c), **bf)
            self.B["d%d" % lvl] = t.empty((N, h, w, c), **bf)
        self.out = t.empty((N, H, W, self.cout), dtype=t.float32, device="cuda")
        # gradient buffers (one per activation shape)
        self.D = {k: t.empty(v.shape, **bf) for k, v in self.B.items()}
        for (h, w, c) in dims:
            self.D["_tmp_%d_%d" % (h, c)] = t.empty((N, h, w, c), **bf)
        self.D["x"] = t.empty((N, H, W, self.cinp), **bf)
        self.D["out"] = t.empty_like(self.out)
        # flipped weights of every layer whose data gradient is wanted (all but the first)
        self.wflip = {n: t.empty(9 * a * b, **bf) for n, a, b, taps in self.specs if taps == 9 and n != "e0a"}
        self.loss = t.zeros(1, dtype=t.float64, device="cuda")
        # partial sums of the parameter gradients, which backward adds up in one order at its end:
        # offset and number per layer (a head with more than 8 outputs has none, its kernel adds).
        # At batch 4 a step takes 0.88 ms, 0.83 with the kernels adding by atomics; adding up after
        # each layer, in memory that stays in L2, 0.95.
        self.parts, used = {}, 0
        for name, a, b, taps in self.specs:
            lvl = 3 if name in ("b_a", "b_b") else 0 if taps == 1 else int(name[1])
            if taps == 9:
                n = self.lib.tpfnet_wgrad_parts(N, H >> lvl, W >> lvl, a, b)
            else:
                n = self.lib.tpfnet_head_parts(N * H * W, a, b)
            if n:
                self.parts[name] = (used, n)
                used += -(-n * (taps * a * b + b) // 128) * 128
        self._part, self._part_words = None, used  # (taken by the first backward pass)
        self._shape = (N, H, W)

    def _chk(self, rc, what):
        if rc != 0:
            raise RuntimeError("tpfnet kernel %s failed (%d)" % (what, rc))

    def _s(self):
        return C.c_void_p(self.stream.cuda_stream)

    # ---------------------------------------------------------- forward
    def forward(self, x):
        """x: bf16 CUDA tensor (N, H, W, cin padded to 32).  Returns float32 (N, H, W, cout)."""
        N, H, W, _ = x.shape
        self._buffers(N, H, W)
        self.x = x
        B, u = self.B, _Net()
        u.cin, u.cout, u.ch = self.cinp, self.cout, self.ch
        names = [n for n, _, _, taps in self.specs if taps == 9]
        u.weight = tuple(self.Pb[n + ".W"].data_ptr() for n in names)
        u.bias = tuple(self.P[n + ".b"].data_ptr() for n in names)
        u.head_w, u.head_b = self.P["head.W"].data_ptr(), self.P["head.b"].data_ptr()
        u.enc = tuple(B[k].data_ptr() for k in ("e0a", "e1a", "e2a", "ba"))
        u.pool = tuple(B["pool%d" % k].data_ptr() for k in (1, 2, 3))
        u.cat = tuple(B["cat%d" % k].data_ptr() for k in (0, 1, 2))
        u.deep = B["b"].data_ptr()
        u.dec_a = tuple(B["d%da" % k].data_ptr() for k in (0, 1, 2))
        u.dec = tuple(B["d%d" % k].data_ptr() for k in (0, 1, 2))
        self._chk(self.lib.tpfnet_unet_forward(C.addressof(u), _p(x), N, H, W, _p(self.out), self._s()), "forward")
        return self.out

    # --------------------------------------------------------- backward
    def _flip_weights(self):
        names = list(self.wflip)
        n = len(names)
        spec = {name: (a, b) for name, a, b, _ in self.specs}
        wt = (_vp * n)(*[self.Pb[k + ".W"].data_ptr() for k in names])
        wf = (_vp * n)(*[self.wflip[k].data_ptr() for k in names])
        ci = (_ip * n)(*[spec[k][0] for k in names])
        co = (_ip * n)(*[spec[k][1] for k in names])
        self._chk(self.lib.tpfnet_flip_weights(n, wt, ci, co, wf, self._s()), "flip")

    def _part_of(self, name):
        return C.c_void_p(self._part.data_ptr() + 4 * self.parts[name][0])

    def _wgrad(self, name, x, dz, N, h, w, cin, c):
        self._chk(self.lib.tpfnet_conv3x3_wgrad_part(_p(x), _p(dz), N, h, w, cin, c, self._part_of(name), self._s()),
                  "wgrad")

    def _sum_parts(self):
        """Adds the partial sums of this backward pass to the gradients."""
        rows = []
        for name, a, b, taps in self.specs:
            if name not in self.parts:
                continue
            at, n = self.parts[name]
            w = taps * a * b
            for key, o, k in ((".W", 0, w), (".b", w, b)):
                rows.append((self._part.data_ptr() + 4 * (at + o), w + b, k, n, self.G[name + key].data_ptr()))
        n = len(rows)
        part, stride, count, parts, dst = ((t * n)(*v) for t, v in zip((_vp, _ll, _ip, _ip, _vp), zip(*rows)))
        self._chk(self.lib.tpfnet_sum_parts(n, part, stride, count, parts, dst, self._s()), "sum_parts")

    def _block_back(self, ka, kb, inp, cin, a, c, dout, dinp, N, h, w):
        """Back through relu(conv_b(relu(conv_a(inp)))): dout (gradient at the block's output,
        its ReLU mask applied) -> weight gradients and dinp (None: not wanted)."""
        L, s = self.lib, self._s()
        da = self.D["_tmp_%d_%d" % (h, c)]
        self._wgrad(kb, a, dout, N, h, w, c, c)
        self._chk(L.tpfnet_conv3x3_dgrad_masked(_p(dout), N, h, w, c, _p(self.wflip[kb]), c, _p(a), _p(da), s), "dgrad")
        self._wgrad(ka, inp, da, N, h, w, cin, c)
        if dinp is not None:
            self._chk(L.tpfnet_conv3x3_dgrad_masked(_p(da), N, h, w, c, _p(self.wflip[ka]), cin, None, _p(dinp), s),
                      "dgrad")

    def backward(self, dout):
        """dout: float32 (N, H, W, cout) gradient of the loss at the output; accumulates
        every parameter gradient into self.G, in the same order on every run.  The ReLU
        masks, the split of the concatenations' gradients and the sums at the encoder's
        outputs are part of the kernels that produce those gradients."""
        L, s = self.lib, self._s()
        N, H, W = self._shape
        if self._part is None:
            with self._on_stream():
                self._part = self.torch.empty(self._part_words, dtype=self.torch.float32, device="cuda")
        B, D = self.B, self.D
        c0, c1, c2, c3 = self.ch
        dims = [(H, W), (H // 2, W // 2), (H // 4, W // 4), (H // 8, W // 8)]
        self._flip_weights()
        if "head" in self.parts:
            rc = L.tpfnet_head_back_part(_p(B["d0"]), _p(dout), N * H * W, c0, _p(self.P["head.W"]), self.cout,
                                         _p(D["d0"]), self._part_of("head"), s)
        else:
            rc = L.tpfnet_head_back_masked(_p(B["d0"]), _p(dout), N * H * W, c0, _p(self.P["head.W"]), self.cout,
                                           _p(D["d0"]), _p(self.G["head.W"]), _p(self.G["head.b"]), s)
        self._chk(rc, "head_back")
        # decoder levels 0, 1, 2; the upsampled part's gradient goes to the level below
        ups = {0: c1, 1: c2, 2: c3}
        skips = {0: c0, 1: c1, 2: c2}
        below = {0: "d1", 1: "d2", 2: "b"}
        for lvl in (0, 1, 2):
            h, w = dims[lvl]
            cu, cs = ups[lvl], skips[lvl]
            ctot = cu + cs
            self._block_back("d%da" % lvl, "d%db" % lvl, B["cat%d" % lvl], ctot, B["d%da" % lvl], cs, D["d%d" % lvl],
                             D["cat%d" % lvl], N, h, w)
            self._chk(L.tpfnet_up_back_masked(_p(D["cat%d" % lvl]), N, h, w, ctot, 0, cu, _p(B[below[lvl]]),
                                              _p(D[below[lvl]]), s), "up_back")
        # bottleneck and encoder levels 2, 1, 0; an encoder output's gradient is the skip part
        # of the concatenation's plus the pooled one's
        for lvl, nm, c in ((3, "b", c3), (2, "e2", c2), (1, "e1", c1)):
            h, w = dims[lvl]
            ka, kb = ("b_a", "b_b") if nm == "b" else (nm + "a", nm + "b")
            pc = self.ch[lvl - 1]
            self._block_back(ka, kb, B["pool%d" % lvl], pc, B[nm + "a"], c, D[nm], D["pool%d" % lvl], N, h, w)
            above = lvl - 1
            skip, act = D["cat%d" % above][..., ups[above]:], B["e%d" % above]
            self._chk(L.tpfnet_pool_back_skip(_p(D["pool%d" % lvl]), N, 2 * h, 2 * w, pc, _p(skip), skip.stride(2),
                                              _p(act), act.stride(2), _p(D["e%d" % above]), s), "pool_back")
        self._block_back("e0a", "e0b", self.x, self.cinp, B["e0a"], c0, D["e0"], None, N, H, W)
        self._sum_parts()

    def zero_grad(self):
        with self._on_stream():
            for g in [self._flat["G"]] if self._is_flat(("G",)) else self.G.values():
                g.zero_()

    def adam(self, lr=1e-3, b1=0.9, b2=0.999, eps=1e-8):
        self.adam_t += 1
        s = self._s()
        if self._is_flat(("P", "G", "M", "V", "Pb")):
            # the 128-element gaps and the biases' unused bf16 copies go along
            f = self._flat
            self._chk(self.lib.tpfnet_adam(_p(f["P"]), _p(f["G"]), _p(f["M"]), _p(f["V"]), f["P"].numel(), lr, b1, b2,
                                           eps, self.adam_t, _p(f["Pb"]), s), "adam")
            return
        for k, p in self.P.items():
            self._chk(self.lib.tpfnet_adam(_p(p), _p(self.G[k]), _p(self.M[k]), _p(self.V[k]), p.numel(), lr, b1, b2,
                                           eps, self.adam_t, _p(self.Pb[k]), s), "adam")

    def mse(self, pred, target, wch=None, want_grad=True):
        """Loss (float, synchronises) and, when want_grad, its gradient in self.D['out']."""
        self._mse(pred, target, wch, want_grad)
        with self._on_stream():
            return float(self.loss.item())

    def _mse(self, pred, target, wch, want_grad=True):
        with self._on_stream():
            self.loss.zero_()
        C_ = pred.shape[-1]
        self._chk(self.lib.tpfnet_mse(_p(pred), _p(target), _p(wch), pred.numel(), C_,
                                      _p(self.D["out"]) if want_grad else None, _p(self.loss), self._s()), "mse")

    def train_step(self, x, target, wch=None, lr=1e-3):
        self.zero_grad()
        out = self.forward(x)
        self._mse(out, target, wch)
        # the loss travels to the host while the backward pass is queued: the GPU does not wait
        # for the host to read it
        t = self.torch
        host = t.empty(1, dtype=t.float64, pin_memory=True)
        done = t.cuda.Event()
        with self._on_stream():
            host.copy_(self.loss, non_blocking=True)
            done.record()
        self.backward(self.D["out"])
        self.adam(lr)
        done.synchronize()
        return float(host)

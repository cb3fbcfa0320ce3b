"""Learned warm start: a 3D convolutional encoder-decoder that predicts the steady velocity and
concentration of the reactive porous-media workload from its geometry and transport numbers.

The lattice Boltzmann step (lbm.py) then starts from the prediction instead of from rest and
relaxes it to its own steady state; its residual, not the network, decides convergence, so a
poor prediction costs steps but never accuracy.  Plain LBM from rest stays the fallback and the
arbiter of the network's error.

Binding: the `lbm_nn_*` functions below carry the C ABI's names (include/lbm_nn.h) and only
marshal torch tensors into device pointers; every operation runs in liblbm.so's sm_103a kernels
(the 3^3 convolutions as implicit GEMMs on the tcgen05 tensor cores, BF16 storage, FP32 accumulation).
PyTorch is used for device memory and the stream only.

Network (the same plan as the FP64 reference of the test suite): encoder levels of two 3^3
convolutions (ReLU) and 2x average pooling, a bottleneck of two 3^3 convolutions, decoder levels
of 2x nearest upsampling, concatenation with the encoder output of that level and one 3^3
convolution (ReLU), and a 1x1 head to 4 outputs.  Inputs (5 channels): solid indicator,
x / (nx - 1), ln(Pe / 10), ln(Da / 0.1) and the distance to the nearest solid over the mean sphere
radius (pore size, which sets how far a pore's concentration is depleted).  Outputs: u / 0.005 (3 channels) and 2 (C - 1/2), which
weights the concentration, the field whose error sets the relaxation time, above the velocity.
Training: masked mean squared error over fluid voxels, Adam.
"""
from __future__ import annotations

import ctypes as C
import math

import numpy as np

from . import lbm as _lbm

U_SCALE = 0.005      # velocity scale of the targets (of the order of the packings' mean fluid speed)
C_OFF, C_SCALE = 0.5, 2.0   # concentration target 2 (C - 1/2): order one, and weighted above u
PE0, DA0 = 10.0, 0.1
OUT_F32, OUT_BF16, OUT_BF16_RELU = 0, 1, 2
PORE_SCALE = 9.0     # length scale of the pore-size channel (the packings' mean sphere radius)
N_FEATURES = 5

_NN = None


def nn_lib():
    """liblbm.so with the lbm_nn_* signatures declared (raises if the library is missing)."""
    global _NN
    if _NN is not None:
        return _NN
    lib = _lbm.load()
    vp, i32, i64, f32 = C.c_void_p, C.c_int32, C.c_int64, C.c_float
    sig = {
        "lbm_nn_gemm_tn": [vp, vp, vp, i64, i32, i32, i32, i32, i32, vp, vp],
        "lbm_nn_status": [vp],
        "lbm_nn_im2col": [vp, vp, i32, i32, i32, i32, i32, i32, vp],
        "lbm_nn_im2col_cv": [vp, vp, i32, i32, i32, i32, i32, vp],
        "lbm_nn_transpose": [vp, vp, i64, i32, vp],
        "lbm_nn_reduce_splits": [vp, vp, i64, i32, i64, vp],
        "lbm_nn_relu_grad": [vp, vp, vp, i64, vp],
        "lbm_nn_pool2": [vp, vp, i32, i32, i32, i32, i32, vp],
        "lbm_nn_up2": [vp, vp, i32, i32, i32, i32, i32, vp],
        "lbm_nn_concat": [vp, i32, vp, i32, vp, i64, i32, vp],
        "lbm_nn_colsum": [vp, vp, i64, i32, vp],
        "lbm_nn_head_fwd": [vp, vp, vp, vp, i64, i32, i32, vp],
        "lbm_nn_head_bwd": [vp, vp, vp, vp, vp, vp, i64, i32, i32, vp],
        "lbm_nn_mse": [vp, vp, vp, vp, vp, i64, i32, i64, vp],
        "lbm_nn_adam": [vp, vp, vp, vp, i64, f32, f32, f32, f32, i32, vp],
        "lbm_nn_pack_weights": [vp, vp, vp, i32, i32, i32, i32, vp],
        "lbm_nn_unpack_wgrad": [vp, vp, i32, i32, vp],
        "lbm_nn_add": [vp, vp, vp, i64, vp],
        "lbm_nn_cast_bf16": [vp, vp, i64, vp],
        "lbm_nn_relu_grad_bias": [vp, vp, vp, vp, vp, i32, i32, i32, i32, vp],
        "lbm_nn_conv3": [vp, i32, i32, vp, i32, i32, i32, i32, vp, i32, vp, i32, vp, i32, vp, vp],
        "lbm_nn_conv3_wgrad": [vp, i32, i32, vp, i32, i32, i32, i32, vp, i32, vp, vp, vp],
        "lbm_nn_conv3_pack": [vp, vp, vp, i32, i32, vp],
        "lbm_nn_pad8": [vp, vp, i64, i32, vp],
    }
    for name, args in sig.items():
        fn = getattr(lib, name)
        fn.argtypes = args
        fn.restype = C.c_int
    lib.lbm_nn_gemm_splits.argtypes = [i32, i32]
    lib.lbm_nn_gemm_splits.restype = i32
    lib.lbm_nn_conv3_packed.argtypes = [i32, i32]
    lib.lbm_nn_conv3_packed.restype = i64
    lib.lbm_nn_conv3_fits.argtypes = [i32, i32, i32, i32]
    lib.lbm_nn_conv3_fits.restype = i32
    lib.lbm_nn_conv3_wgrad_scratch.argtypes = [i32, i32, i32, i32, i32]
    lib.lbm_nn_conv3_wgrad_scratch.restype = i64
    _NN = lib
    return lib


def _p(t):
    return None if t is None else C.c_void_p(t.data_ptr())


def _stream():
    import torch
    return C.c_void_p(torch.cuda.current_stream().cuda_stream)


def _ck(name, st):
    if st != 0:
        raise _lbm.LbmError(st, f"{name} failed")


def _call(name, *args):
    _ck(name, getattr(nn_lib(), name)(*args, _stream()))


# ------------------------------------------------------------------ the C ABI, marshalled

def lbm_nn_gemm_tn(A, B, Cout, ldc, M, N, K, splits=1, out_kind=OUT_F32, bias=None):
    _call("lbm_nn_gemm_tn", _p(A), _p(B), _p(Cout), ldc, M, N, K, splits, out_kind, _p(bias))


def lbm_nn_gemm_splits(K, splits):
    return int(nn_lib().lbm_nn_gemm_splits(K, splits))


def lbm_nn_status():
    _ck("lbm_nn_status", nn_lib().lbm_nn_status(_stream()))


def lbm_nn_im2col(x, col, D, H, W, Cc, Kp, transposed=0):
    _call("lbm_nn_im2col", _p(x), _p(col), D, H, W, Cc, Kp, transposed)


def lbm_nn_im2col_cv(xT, colT, D, H, W, Cc, Kp):
    _call("lbm_nn_im2col_cv", _p(xT), _p(colT), D, H, W, Cc, Kp)


def lbm_nn_transpose(x, y, R, Cc):
    _call("lbm_nn_transpose", _p(x), _p(y), R, Cc)


def lbm_nn_reduce_splits(part, out, n, splits, stride):
    _call("lbm_nn_reduce_splits", _p(part), _p(out), n, splits, stride)


def lbm_nn_relu_grad(y, dy, dx, n):
    _call("lbm_nn_relu_grad", _p(y), _p(dy), _p(dx), n)


def lbm_nn_pool2(i, o, D, H, W, Cc, backward=0):
    _call("lbm_nn_pool2", _p(i), _p(o), D, H, W, Cc, backward)


def lbm_nn_up2(i, o, D, H, W, Cc, backward=0):
    _call("lbm_nn_up2", _p(i), _p(o), D, H, W, Cc, backward)


def lbm_nn_concat(a, Ca, b, Cb, out, V, backward=0):
    _call("lbm_nn_concat", _p(a), Ca, _p(b), Cb, _p(out), V, backward)


def lbm_nn_colsum(x, out, V, Cc):
    _call("lbm_nn_colsum", _p(x), _p(out), V, Cc)


def lbm_nn_head_fwd(h, w, b, y, V, Cc, Co):
    _call("lbm_nn_head_fwd", _p(h), _p(w), _p(b), _p(y), V, Cc, Co)


def lbm_nn_head_bwd(h, w, dy, dh, dw, db, V, Cc, Co):
    _call("lbm_nn_head_bwd", _p(h), _p(w), _p(dy), _p(dh), _p(dw), _p(db), V, Cc, Co)


def lbm_nn_mse(y, t, fluid, dy, loss, V, Co, n_fluid):
    _call("lbm_nn_mse", _p(y), _p(t), _p(fluid), _p(dy), _p(loss), V, Co, n_fluid)


def lbm_nn_adam(w, g, m, v, n, lr, b1, b2, eps, step):
    _call("lbm_nn_adam", _p(w), _p(g), _p(m), _p(v), n, lr, b1, b2, eps, step)


def lbm_nn_pack_weights(w, wk, wt, Co, Ci, Kp, Kpt):
    _call("lbm_nn_pack_weights", _p(w), _p(wk), _p(wt), Co, Ci, Kp, Kpt)


def lbm_nn_unpack_wgrad(dwcol, dw, Co, Ci):
    _call("lbm_nn_unpack_wgrad", _p(dwcol), _p(dw), Co, Ci)


def lbm_nn_add(a, b, y, n):
    _call("lbm_nn_add", _p(a), _p(b), _p(y), n)


def lbm_nn_cast_bf16(x, y, n):
    _call("lbm_nn_cast_bf16", _p(x), _p(y), n)


def lbm_nn_relu_grad_bias(y, dy, dskip, dx, db, shape, Cc):
    _call("lbm_nn_relu_grad_bias", _p(y), _p(dy), _p(dskip), _p(dx), _p(db), *shape, Cc)


def lbm_nn_conv3(src, shape, wp, N, y0, n0, y1=None, bias=None, relu=0):
    """src: (xa, Ca, up, xb, Cb), the input's parts (xb None with Cb 0)."""
    xa, ca, up, xb, cb = src
    _call("lbm_nn_conv3", _p(xa), ca, up, _p(xb), cb, *shape, _p(wp), N, _p(bias), relu, _p(y0), n0, _p(y1))


def lbm_nn_conv3_wgrad(src, shape, dy, Co, scratch, dw):
    xa, ca, up, xb, cb = src
    _call("lbm_nn_conv3_wgrad", _p(xa), ca, up, _p(xb), cb, *shape, _p(dy), Co, _p(scratch), _p(dw))


def lbm_nn_conv3_wgrad_scratch(shape, Cc, Co):
    return int(nn_lib().lbm_nn_conv3_wgrad_scratch(*shape, Cc, Co))


def lbm_nn_pad8(x, x8, V, Cc):
    _call("lbm_nn_pad8", _p(x), _p(x8), V, Cc)


def lbm_nn_conv3_pack(w, wp, wtp, Co, Ci):
    _call("lbm_nn_conv3_pack", _p(w), _p(wp), _p(wtp), Co, Ci)


def lbm_nn_conv3_packed(Co, Ci):
    return int(nn_lib().lbm_nn_conv3_packed(Co, Ci))


def lbm_nn_conv3_fits(Ca, up, Cb, Co):
    return bool(nn_lib().lbm_nn_conv3_fits(Ca, up, Cb, Co))


# ------------------------------------------------------------------ network

def kpad(k):
    """K of a 3^3 convolution padded to the GEMM's 128-row tiles."""
    return ((k + 127) // 128) * 128


def layer_plan(c_in=4, c_out=4, width=(16, 32, 64, 160)):
    """(name, kind, C_in, C_out) of every convolution, in forward order."""
    plan, c = [], c_in
    for l, wd in enumerate(width[:-1]):
        plan += [(f"enc{l}a", "conv3", c, wd), (f"enc{l}b", "conv3", wd, wd)]
        c = wd
    plan += [("mid_a", "conv3", c, width[-1]), ("mid_b", "conv3", width[-1], width[-1])]
    c = width[-1]
    for l in reversed(range(len(width) - 1)):
        plan.append((f"dec{l}", "conv3", c + width[l], width[l]))
        c = width[l]
    plan.append(("head", "conv1", c, c_out))
    return plan


class WarmStartNet:
    """The encoder-decoder on one GPU: FP32 master weights with Adam, BF16 copies for the
    tensor-core GEMMs, channel-last BF16 activations."""

    def __init__(self, width=(16, 32, 64, 160), c_in=N_FEATURES, c_out=4, seed=0, device=0):
        import torch
        if width[0] != 16 or c_out != 4:
            raise ValueError("the head kernel takes 16 input and 4 output channels")
        if any(w % 16 for w in width):
            raise ValueError("channel widths must be multiples of 16 (GEMM N tiles)")
        self.torch = torch
        self.dev = torch.device("cuda", device)
        self.width, self.c_in, self.c_out = tuple(width), c_in, c_out
        self.plan = layer_plan(c_in, c_out, width)
        self.L = len(width) - 1
        # one flat FP32 buffer of parameters (views per tensor), gradients and Adam moments
        shapes = {}
        for name, kind, ci, co in self.plan:
            shapes[name + ".w"] = (co, ci, 27) if kind == "conv3" else (co, ci)
            shapes[name + ".b"] = (co,)
        self.shapes = shapes
        n = sum(int(np.prod(s)) for s in shapes.values())
        self.n_params = n
        f32 = dict(dtype=torch.float32, device=self.dev)
        self.flat = torch.zeros(n, **f32)
        self.gflat = torch.zeros(n, **f32)
        self.m = torch.zeros(n, **f32)
        self.v = torch.zeros(n, **f32)
        self.p, self.g, off = {}, {}, 0
        for k, s in shapes.items():
            sz = int(np.prod(s))
            self.p[k] = self.flat[off:off + sz].view(s)
            self.g[k] = self.gflat[off:off + sz].view(s)
            off += sz
        rng = np.random.default_rng(seed)
        init = {}
        for name, kind, ci, co in self.plan:
            fan = ci * (27 if kind == "conv3" else 1)
            init[name + ".w"] = rng.standard_normal(shapes[name + ".w"]) * math.sqrt(2.0 / fan)
            init[name + ".b"] = np.zeros(co)
        self.set_params(init)
        self.step_count = 0
        self._scratch = None

    # -------------------------------------------------------------- parameters

    def set_params(self, params):
        """Load parameters given as numpy arrays (conv weights [Co, Ci, 3, 3, 3] or [Co, Ci, 27],
        head [Co, Ci], biases [Co]) and repack the BF16 GEMM copies."""
        for k, v in params.items():
            self.p[k].copy_(self.torch.from_numpy(np.asarray(v, np.float32).reshape(self.shapes[k])))
        self._pack()

    def params_numpy(self):
        return {k: v.detach().cpu().numpy().copy() for k, v in self.p.items()}

    def grads_numpy(self):
        return {k: v.detach().cpu().numpy().copy() for k, v in self.g.items()}

    def _pack(self):
        """BF16 operands of the 3^3 kernels: wp for the convolution, wt (flipped, transposed) for its
        input gradient; layers that lbm_nn_conv3 does not take get the im2col GEMM's."""
        torch = self.torch
        if not hasattr(self, "wp"):
            bf = dict(dtype=torch.bfloat16, device=self.dev)
            self.wp, self.wt, self.rows = {}, {}, {}
            for name, kind, ci, co in self.plan:
                if kind != "conv3":
                    continue
                cb = self.width[int(name[3])] if name.startswith("dec") else 0
                self.rows[name] = not lbm_nn_conv3_fits(ci - cb, cb > 0, cb, co)
                if self.rows[name]:
                    self.wp[name] = torch.empty((co, kpad(27 * ci)), **bf)
                    self.wt[name] = torch.empty((ci, kpad(27 * co)), **bf)
                else:
                    self.wp[name] = torch.empty(lbm_nn_conv3_packed(co, ci), **bf)
                    self.wt[name] = torch.empty(lbm_nn_conv3_packed(ci, co), **bf) if ci % 16 == 0 else None
        for name, kind, ci, co in self.plan:
            if kind != "conv3":
                continue
            if self.rows[name]:
                lbm_nn_pack_weights(self.p[name + ".w"], self.wp[name], self.wt[name], co, ci, kpad(27 * ci), kpad(27 * co))
            else:
                lbm_nn_conv3_pack(self.p[name + ".w"], self.wp[name], self.wt[name], co, ci)

    # -------------------------------------------------------------- layers
    # An input is (xa, Ca, up, xb, Cb): one tensor, or the decoder's pair of a coarse tensor, upsampled as it is
    # read, and the encoder's output of the level.

    def _empty(self, rows, cols, dtype=None):
        return self.torch.empty((rows, cols), dtype=dtype or self.torch.bfloat16, device=self.dev)

    def _scratch_for(self, n):
        if self._scratch is None or self._scratch.numel() < n:
            self._scratch = self.torch.empty(n, dtype=self.torch.float32, device=self.dev)
        return self._scratch

    def _conv3(self, name, src, shape, co):
        V = shape[0] * shape[1] * shape[2]
        if V % 128:
            raise _lbm.LbmError(-1, f"{name}: the number of voxels must be a multiple of 128")
        y = self._empty(V, co)
        if self.rows[name]:
            x, ci = self._joined(src, shape)
            kp = kpad(27 * ci)
            col = self._empty(V, kp)
            lbm_nn_im2col(x, col, *shape, ci, kp, 0)
            lbm_nn_gemm_tn(col, self.wp[name], y, co, V, co, kp, 1, OUT_BF16_RELU, self.p[name + ".b"])
        else:
            lbm_nn_conv3(src, shape, self.wp[name], co, y, co, bias=self.p[name + ".b"], relu=1)
        return y

    def _conv3_backward(self, name, src, yout, dy, dskip, shape, co, need_dx=True):
        """Gradients of a layer's weights and bias from dy (with dskip: dy is the gradient of the pooled
        output and dskip the skip connection's); returns those of the parts of its input."""
        V = shape[0] * shape[1] * shape[2]
        _, ca, _, _, cb = src
        dpre = self._empty(V, co)
        lbm_nn_relu_grad_bias(yout, dy, dskip, dpre, self.g[name + ".b"], shape, co)
        if self.rows[name]:
            return self._rows_backward(name, src, dpre, shape, co, need_dx)
        lbm_nn_conv3_wgrad(src, shape, dpre, co, self._scratch_for(lbm_nn_conv3_wgrad_scratch(shape, ca + cb, co)),
                           self.g[name + ".w"])
        if not need_dx:
            return None, None
        # input gradient: a convolution of dpre with the flipped, transposed kernel
        da, db = self._empty(V, ca), self._empty(V, cb) if cb else None
        lbm_nn_conv3((dpre, co, 0, None, 0), shape, self.wt[name], ca + cb, da, ca, db)
        return da, db

    # Layers outside lbm_nn_conv3's range (an input of 9 or more channels that is no multiple of 16, very wide
    # layers): im2col rows and plain GEMMs.

    def _joined(self, src, shape):
        xa, ca, up, xb, cb = src
        if not cb:
            return xa, ca
        D, H, W = shape
        fine = self._empty(D * H * W, ca)
        lbm_nn_up2(xa, fine, D // 2, H // 2, W // 2, ca, 0)
        cat = self._empty(D * H * W, ca + cb)
        lbm_nn_concat(fine, ca, xb, cb, cat, D * H * W, 0)
        return cat, ca + cb

    def _rows_backward(self, name, src, dpre, shape, co, need_dx):
        D, H, W = shape
        V = D * H * W
        _, ca, _, _, cb = src
        x, ci = self._joined(src, shape)
        kp, kpt = kpad(27 * ci), kpad(27 * co)
        # weight gradient: dW[k][o] = sum_v colT[k][v] dpreT[o][v], split over v; colT is built
        # from a channel-major copy of the input when the rows allow 8-voxel vectors
        col = self._empty(kp, V)
        if W % 8 == 0:
            xT = self._empty(ci, V)
            lbm_nn_transpose(x, xT, V, ci)
            lbm_nn_im2col_cv(xT, col, D, H, W, ci, kp)
        else:
            lbm_nn_im2col(x, col, D, H, W, ci, kp, 1)
        dpreT = self._empty(co, V)
        lbm_nn_transpose(dpre, dpreT, V, co)
        tiles = (kp // 128) * max(1, co // 128)
        splits = lbm_nn_gemm_splits(V, max(1, min(64, (4 * 152) // max(1, tiles), V // 64)))
        part = self._scratch_for(splits * kp * co)
        lbm_nn_gemm_tn(col, dpreT, part, co, kp, co, V, splits, OUT_F32, None)
        dwcol = self._empty(kp, co, self.torch.float32)
        lbm_nn_reduce_splits(part, dwcol, kp * co, splits, kp * co)
        lbm_nn_unpack_wgrad(dwcol, self.g[name + ".w"], co, ci)
        if not need_dx:
            return None, None
        col = self._empty(V, kpt)
        lbm_nn_im2col(dpre, col, D, H, W, co, kpt, 0)
        dx = self._empty(V, ci)
        lbm_nn_gemm_tn(col, self.wt[name], dx, ci, V, ci, kpt, 1, OUT_BF16, None)
        if not cb:
            return dx, None
        da, db = self._empty(V, ca), self._empty(V, cb)
        lbm_nn_concat(da, ca, db, cb, dx, V, 1)
        return da, db

    # -------------------------------------------------------------- passes

    def forward(self, x, shape):
        """x: BF16 [V][c_in] channel-last; returns FP32 [V][c_out] and keeps the activations."""
        # per layer: its input, its output and the sizes
        acts = {}
        h, shp, c = x, tuple(shape), self.c_in
        if not self.rows["enc0a"] and c <= 8:   # the narrow input, in rows of 8 channels
            h = self._empty(shp[0] * shp[1] * shp[2], 8)
            lbm_nn_pad8(x, h, h.shape[0], c)
        skips = []
        for l, wd in enumerate(self.width[:-1]):
            for s in "ab":
                n, src = f"enc{l}{s}", (h, c, 0, None, 0)
                h = self._conv3(n, src, shp, wd)
                c = wd
                acts[n] = (src, h, shp)
            skips.append((h, shp, c))
            D, H, W = shp
            shp = (D // 2, H // 2, W // 2)
            pooled = self._empty(shp[0] * shp[1] * shp[2], c)
            lbm_nn_pool2(h, pooled, D, H, W, c, 0)
            h = pooled
        for n in ("mid_a", "mid_b"):
            src = (h, c, 0, None, 0)
            h = self._conv3(n, src, shp, self.width[-1])
            c = self.width[-1]
            acts[n] = (src, h, shp)
        for l in reversed(range(self.L)):
            sk, shp, sc = skips[l]
            n, src = f"dec{l}", (h, c, 1, sk, sc)
            h = self._conv3(n, src, shp, self.width[l])
            c = self.width[l]
            acts[n] = (src, h, shp)
        V = shp[0] * shp[1] * shp[2]
        y = self._empty(V, self.c_out, self.torch.float32)
        lbm_nn_head_fwd(h, self.p["head.w"], self.p["head.b"], y, V, c, self.c_out)
        self._acts = acts
        return y

    def backward(self, dy):
        """dy: FP32 [V][c_out] = dL/dy of the last forward; fills the gradients."""
        acts = self._acts
        _, h, shp = acts["dec0"]
        V, c = h.shape
        dh = self._empty(V, c)
        lbm_nn_head_bwd(h, self.p["head.w"], dy, dh, self.g["head.w"], self.g["head.b"], V, c, self.c_out)
        dskip = {}
        for l in range(self.L):
            src, y, (D, H, W) = acts[f"dec{l}"]
            du, dskip[l] = self._conv3_backward(f"dec{l}", src, y, dh, None, (D, H, W), self.width[l])
            dh = self._empty(D * H * W // 8, src[1])
            lbm_nn_up2(du, dh, D // 2, H // 2, W // 2, src[1], 1)
        for n in ("mid_b", "mid_a"):
            src, y, shp = acts[n]
            dh, _ = self._conv3_backward(n, src, y, dh, None, shp, self.width[-1])
        for l in reversed(range(self.L)):
            # the pooling's gradient and the skip connection's meet in the layer's ReLU gradient
            src, y, shp = acts[f"enc{l}b"]
            dh, _ = self._conv3_backward(f"enc{l}b", src, y, dh, dskip[l], shp, self.width[l])
            src, y, shp = acts[f"enc{l}a"]
            dh, _ = self._conv3_backward(f"enc{l}a", src, y, dh, None, shp, self.width[l], need_dx=l > 0)

    def loss_and_grad(self, y, t, fluid, n_fluid):
        torch = self.torch
        V = y.shape[0]
        dy = torch.empty_like(y)
        loss = torch.zeros(1, dtype=torch.float64, device=self.dev)
        lbm_nn_mse(y, t, fluid, dy, loss, V, self.c_out, n_fluid)
        return loss, dy

    def adam(self, lr=1e-3, b1=0.9, b2=0.999, eps=1e-8):
        self.step_count += 1
        lbm_nn_adam(self.flat, self.gflat, self.m, self.v, self.n_params, lr, b1, b2, eps, self.step_count)
        self._pack()

    def train_step(self, x, t, fluid, n_fluid, shape, lr=1e-3):
        y = self.forward(x, shape)
        loss, dy = self.loss_and_grad(y, t, fluid, n_fluid)
        self.backward(dy)
        self.adam(lr)
        return loss

    def check(self):
        """Raises if a GEMM gave up waiting on its copies since the last check."""
        lbm_nn_status()


# ------------------------------------------------------------------ data

def pore_distance(geom, pad=16):
    """Euclidean distance of every fluid node to the nearest solid node (0 on solids), with the
    domain wrapped periodically in y and z and open in x (inlet and outlet faces)."""
    from scipy.ndimage import distance_transform_edt
    fl = geom == 0
    p = min(pad, geom.shape[0], geom.shape[1])
    big = np.pad(fl, ((p, p), (p, p), (0, 0)), mode="wrap")
    d = distance_transform_edt(big)
    return d[p:p + geom.shape[0], p:p + geom.shape[1], :]


def features(geom, Pe=PE0, Da=DA0, device=0):
    """Input channels (channel-last BF16 [V][5]) of a geometry [nz, ny, nx] of flags: solid
    indicator, x / (nx - 1), ln(Pe / 10), ln(Da / 0.1), distance to the nearest solid / 9."""
    import torch
    nz, ny, nx = geom.shape
    f = np.empty((nz, ny, nx, N_FEATURES), np.float32)
    f[..., 0] = (geom != 0)
    f[..., 1] = (np.arange(nx) / max(1, nx - 1))[None, None, :]
    f[..., 2] = math.log(Pe / PE0)
    f[..., 3] = math.log(Da / DA0)
    f[..., 4] = pore_distance(geom) / PORE_SCALE
    return torch.from_numpy(f.reshape(-1, N_FEATURES)).to(device=torch.device("cuda", device), dtype=torch.bfloat16)


def targets(u, Cf, device=0):
    """Training targets (FP32 [V][4]): u / U_SCALE and C_SCALE (C - C_OFF)."""
    import torch
    nz, ny, nx = Cf.shape[-3:]
    t = np.empty((nz, ny, nx, 4), np.float32)
    for a in range(3):
        t[..., a] = u[a] / U_SCALE
    t[..., 3] = C_SCALE * (Cf.reshape(nz, ny, nx) - C_OFF)
    return torch.from_numpy(t.reshape(-1, 4)).to(torch.device("cuda", device))


def predict_fields(net, geom, Pe=PE0, Da=DA0):
    """(rho, u, C) for lbm Solver.set_fields from the network's prediction: rho = 1, u and C
    from the outputs on fluid nodes (solid nodes: u = 0, C = 1)."""
    import torch
    nz, ny, nx = geom.shape
    with torch.no_grad():
        y = net.forward(features(geom, Pe, Da, net.dev.index), geom.shape)
    net.check()
    y = y.cpu().numpy().reshape(nz, ny, nx, 4)
    fl = geom == 0
    u = np.stack([np.where(fl, y[..., a] * U_SCALE, 0.0) for a in range(3)])
    Cf = np.where(fl, y[..., 3] / C_SCALE + C_OFF, 1.0)[None]
    rho = np.ones((1, nz, ny, nx))
    return rho, u, Cf

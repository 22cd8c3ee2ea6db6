"""Layer and network runners on top of the C-ABI binding (orchestration only).

A layer owns a packed weight handle and a device bias; a network is the list of calls the
C3D-shaped and R(2+1)D-shaped forward passes make (Section 5 of the paper names the
models; pooling / residual structure follows the cited architectures).  Every numerical
step is a call into librt3d; torch provides device memory and streams.
"""
from __future__ import annotations

import contextlib
import dataclasses
import itertools

import numpy as np
import torch

from . import binding as B

_pycall, _ADDRESS = B.pycall(), B.ADDRESS
# The binding's compute functions as they are: calls go round them only while they are what the binding's module holds (a
# tracer or a test that wraps them sees every call).
_FUNCTIONS = {fn: getattr(B, fn) for fn in ("rt3d_conv3d_sparse", "rt3d_conv3d_dense", "rt3d_conv3d_sparse_fused",
                                            "rt3d_conv2plus1d_fused", "rt3d_maxpool3d", "rt3d_add_relu", "rt3d_copy_f32")}


def _unwrapped(*names) -> bool:
    return B.noting() is None and all(getattr(B, fn) is _FUNCTIONS[fn] for fn in names)


def pitch_for(c: int, dtype) -> int:
    """Channel pitch that satisfies the library's alignment rule (16 bytes per voxel row start)."""
    mult = 8 if dtype == torch.bfloat16 else 4
    return -(-c // mult) * mult


def to_device(x_np: np.ndarray, dtype=torch.bfloat16, c_stride: int | None = None, device="cuda"):
    """float32 numpy NDHWC -> device tensor [n,t,h,w,c_stride] (extra channels zero)."""
    c = x_np.shape[-1]
    cs = pitch_for(c, dtype) if c_stride is None else c_stride
    t = torch.zeros(x_np.shape[:-1] + (cs,), dtype=dtype, device=device)
    t[..., :c] = torch.from_numpy(np.ascontiguousarray(x_np)).to(dtype).to(device)
    return t


def to_numpy(t: torch.Tensor, c: int) -> np.ndarray:
    return t[..., :c].float().cpu().numpy()


# The last assignment to any layer's attribute, a value of its own for each: a noted sequence of calls holds from one to the next.
_changes, _layer_changes = itertools.count(1), 0


class ConvLayer:
    """One convolution layer: packed weights (KGS mask or dense) + bias on the device."""

    def __setattr__(self, name, value):
        global _layer_changes
        object.__setattr__(self, name, value)
        object.__setattr__(self, "_params", {})     # parameter structures by (ReLU, kernel family, zero padding, concurrent)
        _layer_changes = next(_changes)

    def __init__(self, spec, w, bias, mask, g_m=4, g_n=4, dtype=torch.bfloat16, dense=False, device="cuda"):
        self.spec = spec
        self.dtype = dtype
        cd = B.RT3D_BF16 if dtype == torch.bfloat16 else B.RT3D_F32
        self.dense = dense
        self.packed = B.rt3d_pack_dense(w, cd) if dense else B.rt3d_pack_kgs(w, mask, g_m, g_n, cd)
        self.bias = None if bias is None else torch.from_numpy(np.ascontiguousarray(bias, np.float32)).to(device)
        self.device = device

    def _param_struct(self, relu, algo, x_pad_zero):
        relu = self.spec.relu if relu is None else relu
        key = (relu, algo, x_pad_zero, B.concurrent())
        p = self._params.get(key)
        if p is None:
            p = self._params[key] = B._params(self.spec.stride, self.spec.pad, relu, algo, x_pad_zero)
        return p

    def out_shape(self, x: torch.Tensor):
        n, t, h, w, _ = x.shape
        to, ho, wo = self.spec.out_extent(t, h, w)
        return (n, to, ho, wo, pitch_for(self.spec.cout, self.dtype))

    def alloc_out(self, x: torch.Tensor) -> torch.Tensor:
        return torch.zeros(self.out_shape(x), dtype=self.dtype, device=x.device)

    def __call__(self, x: torch.Tensor, y: torch.Tensor | None = None, algo=B.ALGO_AUTO, relu=None, stream=None,
                 x_pad_zero=False):
        """x_pad_zero: the channels of x beyond spec.cin are known to hold zeros (true for tensors made by
        `to_device`); lets the first-layer kernel fetch whole image rows per request."""
        if y is None:
            y = self.alloc_out(x)
        name = "rt3d_conv3d_dense" if self.dense else "rt3d_conv3d_sparse"
        if not _unwrapped(name):
            fn = B.rt3d_conv3d_dense if self.dense else B.rt3d_conv3d_sparse
            fn(B.tensor_desc(x, self.spec.cin), self.packed, self.bias, B.tensor_desc(y, self.spec.cout), self.spec.stride,
               self.spec.pad, self.spec.relu if relu is None else relu, algo, stream, x_pad_zero)
            return y
        status = _pycall.conv(_ADDRESS[name], x, self.spec.cin, self.packed.handle.value, self.bias,
                              self._param_struct(relu, algo, x_pad_zero), y, self.spec.cout, stream)
        if status != B.OK:
            raise B.Rt3dError(status, name)
        return y

    def run_desc(self, xd, yd, algo=B.ALGO_AUTO, stream=None):
        """Same call on ready-made descriptors (e.g. a channel slice of a concatenation buffer as output)."""
        fn = B.rt3d_conv3d_dense if self.dense else B.rt3d_conv3d_sparse
        fn(xd, self.packed, self.bias, yd, self.spec.stride, self.spec.pad, self.spec.relu, algo, stream)

    def fused(self, x: torch.Tensor, y: torch.Tensor, residual: torch.Tensor | None = None, pool=(1, 1, 1),
              relu=None, algo=B.ALGO_AUTO, stream=None, x_pad_zero=False):
        """y = pool(act(conv(x) + bias + residual)) in one launch (rt3d_conv3d_sparse_fused)."""
        if not _unwrapped("rt3d_conv3d_sparse_fused"):
            res = None if residual is None else B.tensor_desc(residual, self.spec.cout)
            B.rt3d_conv3d_sparse_fused(B.tensor_desc(x, self.spec.cin), self.packed, self.bias,
                                       B.tensor_desc(y, self.spec.cout), self.spec.stride, self.spec.pad,
                                       self.spec.relu if relu is None else relu, res, pool, algo, stream, x_pad_zero)
            return y
        status = _pycall.conv(_ADDRESS["rt3d_conv3d_sparse_fused"], x, self.spec.cin, self.packed.handle.value, self.bias,
                              self._param_struct(relu, algo, x_pad_zero), y, self.spec.cout, stream, residual, pool)
        if status != B.OK:
            raise B.Rt3dError(status, "rt3d_conv3d_sparse_fused")
        return y

    def cost(self, x: torch.Tensor):
        return B.rt3d_conv3d_cost(B.tensor_desc(x, self.spec.cin), self.packed, self.spec.stride, self.spec.pad)


def maxpool(x: torch.Tensor, c: int, pool, y: torch.Tensor | None = None, stream=None) -> torch.Tensor:
    n, t, h, w, cs = x.shape
    ext = [(d + 2 * p - k) // s + 1 for d, p, k, s in zip((t, h, w), pool.pad, pool.k, pool.stride)]
    if y is None:
        y = torch.zeros((n, ext[0], ext[1], ext[2], cs), dtype=x.dtype, device=x.device)
    B.rt3d_maxpool3d(B.tensor_desc(x, c), pool.k, pool.stride, pool.pad, B.tensor_desc(y, c), stream)
    return y


def add_relu(a: torch.Tensor, b: torch.Tensor, c: int, relu=True, y: torch.Tensor | None = None, stream=None):
    if y is None:
        y = torch.zeros_like(a)
    B.rt3d_add_relu(B.tensor_desc(a, c), B.tensor_desc(b, c), relu, B.tensor_desc(y, c), stream)
    return y


class Workspace:
    """Activation buffers keyed by (name, shape): allocated on first use, reused afterwards so a
    steady-state forward pass allocates nothing."""

    def __init__(self):
        self.bufs = {}

    def get(self, name, shape, dtype, device):
        key = (name, tuple(shape), dtype)
        if key not in self.bufs:
            self.bufs[key] = torch.zeros(shape, dtype=dtype, device=device)
        return self.bufs[key]


def _record(stream) -> torch.cuda.Event:
    """Event after the work that `stream` holds."""
    ev = torch.cuda.Event()
    ev.record(stream)
    if B.noting() is not None:
        B.noting().note_event(B.CALL_RECORD, stream, ev)
    return ev


def _wait(stream, ev):
    stream.wait_event(ev)
    if B.noting() is not None:
        B.noting().note_event(B.CALL_WAIT, stream, ev)


class _NotedForward:
    """Base of the networks.  The calls of a forward pass are noted when an input of its shape is seen first, and issued
    by one library call from then on (R(2+1)D: 33 calls, 590 us of Python; S3D with every convolution a call
    of its own: 90 calls and 36 stream events, 1730 us).
    Noted passes are dropped when a layer, the memory of a bias or of the output, a switch of the network or its set of
    buffers has changed since."""

    _SWITCHES = ()          # attributes that decide which calls a pass makes
    _MOST = 8               # input shapes remembered

    def _state(self):
        return [getattr(self, name) for name in self._SWITCHES]

    def forward(self, x: torch.Tensor, algo=B.ALGO_AUTO, keep=None, stream=None, **kw) -> torch.Tensor:
        if keep is not None or any(v is not None for v in kw.values()) or B.is_planning() or not _unwrapped(*_FUNCTIONS):
            return self._forward(x, algo, keep, stream, **kw)
        noted = self.__dict__.setdefault("_noted", {})
        # torch.Size, dtype and device hash by value; the current device and whether a stream is named decide the streams
        key = (x.shape, x.stride(), x.dtype, x.device, algo, stream is None, B.concurrent(), torch.cuda.current_device())
        ptr = x.data_ptr()
        found = noted.get(key)
        if found is not None:
            seq, out, buffers, changes, layers, state = found
            if changes == _layer_changes and layers == self._all_layers() and state == self._state() and ptr not in buffers and \
                    seq.holds():
                status = seq.run(ptr, B.current_stream_ptr() if stream is None else int(stream))
                if status == B.OK:
                    return out
            del noted[key]
        seq = B.CallSequence(ptr, B.current_stream_ptr() if stream is None else int(stream))
        changes = _layer_changes
        with seq.noting():
            out = self._forward(x, algo, None, stream)
        buffers = {b.data_ptr(): b for b in self.ws.bufs.values()}      # kept alive as long as the noted calls
        if ptr not in buffers:
            seq.finish(out, buffers.values())
            if len(noted) >= self._MOST:
                noted.pop(next(iter(noted)))
            noted[key] = (seq, out, buffers, changes, self._all_layers(), self._state())
        return out


class C3DNet(_NotedForward):
    """C3D-shaped forward: 8 convs (3x3x3, ReLU) and 5 max-pools.  `layers` maps conv name -> ConvLayer."""

    _SWITCHES = ("plan", "fuse_pool", "input_pad_zero", "ws")

    def _all_layers(self):
        return [*self.layers.values(), *(self.fc_layers or ())]

    def __init__(self, plan, layers, fuse_pool: bool = False, input_pad_zero: bool = True, fc_layers=None):
        self.plan = plan
        self.layers = layers
        self.fc_layers = fc_layers      # optional list of dense 1x1x1 ConvLayer (fc6, fc7, fc8) run on the flattened pool5 block
        self.fuse_pool = fuse_pool      # conv + ReLU + un-padded 2-wide max-pool in one launch where the library can
        self.input_pad_zero = input_pad_zero    # the clip tensor comes from to_device(): channels 3..7 are zeros
        self.ws = Workspace()
        self.fused_ok = {}              # conv name -> did the fused call apply (decided on first use per shape)

    def _try_fused(self, op, pool, x, algo, stream, x_pad_zero=False):
        """Runs conv `op` with `pool` fused; returns the pooled tensor or None if the library declines."""
        if any(pool.pad) or tuple(pool.k) != tuple(pool.stride) or any(k not in (1, 2) for k in pool.k):
            return None
        key = (op.name, tuple(x.shape))
        if self.fused_ok.get(key) is False:
            return None
        layer = self.layers[op.name]
        n, t, h, w, _ = x.shape
        to, ho, wo = op.out_extent(t, h, w)
        shape = (n, to // pool.k[0], ho // pool.k[1], wo // pool.k[2], pitch_for(op.cout, x.dtype))
        y = self.ws.get(pool.name, shape, x.dtype, x.device)
        try:
            layer.fused(x, y, pool=pool.k, algo=algo, stream=stream, x_pad_zero=x_pad_zero)
        except B.Rt3dError as e:
            if e.status != B.ERR_UNSUPPORTED:
                raise
            self.fused_ok[key] = False
            return None
        self.fused_ok[key] = True
        return y

    def forward(self, x: torch.Tensor, algo=B.ALGO_AUTO, keep=None, stream=None, plan_log=None) -> torch.Tensor:
        """plan_log: dict that receives, per conv name, how the library ran that layer (rt3d_last_plan)."""
        return super().forward(x, algo, keep, stream, plan_log=plan_log)

    def _forward(self, x, algo, keep, stream, plan_log=None):
        c = self.plan[0].cin
        skip = None
        for i, op in enumerate(self.plan):
            if op is skip:
                continue
            if hasattr(op, "cout"):
                pad0 = self.input_pad_zero and i == 0
                nxt = self.plan[i + 1] if i + 1 < len(self.plan) else None
                if self.fuse_pool and nxt is not None and not hasattr(nxt, "cout"):
                    y = self._try_fused(op, nxt, x, algo, stream, pad0)
                    if y is not None:
                        if plan_log is not None:
                            plan_log[op.name] = B.rt3d_last_plan()
                        x, c, skip = y, op.cout, nxt
                        if keep is not None:
                            keep[nxt.name] = x
                        continue
                layer = self.layers[op.name]
                y = self.ws.get(op.name, layer.out_shape(x), x.dtype, x.device)
                x = layer(x, y, algo=algo, stream=stream, x_pad_zero=pad0)
                if plan_log is not None:
                    plan_log[op.name] = B.rt3d_last_plan()
                c = op.cout
            else:
                n, t, h, w, cs = x.shape
                ext = [(d + 2 * p - k) // s + 1 for d, p, k, s in zip((t, h, w), op.pad, op.k, op.stride)]
                y = self.ws.get(op.name, (n, ext[0], ext[1], ext[2], cs), x.dtype, x.device)
                x = maxpool(x, c, op, y, stream=stream)
            if keep is not None:
                keep[op.name] = x
        if self.fc_layers:
            x = self.fc_tail(x, c, algo=algo, keep=keep, stream=stream)
        return x

    def fc_tail(self, feat: torch.Tensor, c: int, algo=B.ALGO_AUTO, keep=None, stream=None) -> torch.Tensor:
        """Fully connected layers as 1x1x1 convolutions over the flattened feature block (memory order t, h, w, c;
        needs the block stored without channel padding)."""
        n, t, h, w, cs = feat.shape
        if cs != c:
            raise ValueError("the feature block must have no channel padding to be flattened in place")
        x = feat.view(n, 1, 1, 1, t * h * w * c)
        for layer in self.fc_layers:
            y = self.ws.get(layer.spec.name, layer.out_shape(x), x.dtype, x.device)
            x = layer(x, y, algo=algo, stream=stream)
            if keep is not None:
                keep[layer.spec.name] = x
        return x

    def n_launches(self) -> int:
        return len(self.plan)


class R2Plus1DNet(_NotedForward):
    """R(2+1)D-18-shaped forward: stem, then residual blocks of two factorised convs each
    (spatial 1x3x3 then temporal 3x1x1), optional 1x1x1 strided projection, add + ReLU."""

    _SWITCHES = ("stem", "blocks", "fuse_residual", "fuse_pairs", "ws")

    def _all_layers(self):
        return list(self.layers.values())

    def __init__(self, stem, blocks, layers, fuse_residual: bool = False, fuse_pairs: bool = False):
        self.stem, self.blocks, self.layers = stem, blocks, layers
        self.fuse_residual = fuse_residual      # block end = one fused launch instead of conv + add kernel
        # spatial conv + temporal conv of a factorised pair in ONE launch (rt3d_conv2plus1d_fused) wherever the
        # library takes the pair; the wide intermediate tensor then never reaches device memory.  Needs
        # fuse_residual (the block's second pair ends in the residual add) and is skipped while `keep` collects
        # every layer's output.
        self.fuse_pairs = fuse_pairs and fuse_residual
        self.pairs_fused, self.pairs_declined = set(), set()
        self.side = None
        self.ws = Workspace()

    def _pair(self, s_spec, t_spec, x, residual, relu_t, stream, out_name):
        """The pair in one launch; None if the library declines it (remembered, so it is asked only once)."""
        if s_spec.name in self.pairs_declined or s_spec.stride != (1, 1, 1) or t_spec.stride != (1, 1, 1):
            return None
        ls, lt = self.layers[s_spec.name], self.layers[t_spec.name]
        n, t, h, w, _ = x.shape
        t, h, w = t_spec.out_extent(*s_spec.out_extent(t, h, w))
        y = self.ws.get(out_name, (n, t, h, w, pitch_for(t_spec.cout, x.dtype)), x.dtype, x.device)
        try:
            B.rt3d_conv2plus1d_fused(B.tensor_desc(x, s_spec.cin), ls.packed, ls.bias, s_spec.pad, s_spec.relu, lt.packed,
                                     lt.bias, t_spec.pad, relu_t, B.tensor_desc(y, t_spec.cout),
                                     residual=None if residual is None else B.tensor_desc(residual, t_spec.cout),
                                     stream=stream)
        except B.Rt3dError as e:
            if e.status != B.ERR_UNSUPPORTED:
                raise
            self.pairs_declined.add(s_spec.name)
            return None
        self.pairs_fused.add(s_spec.name)
        return y

    def _conv(self, spec, x, algo, stream):
        layer = self.layers[spec.name]
        y = self.ws.get(spec.name, layer.out_shape(x), x.dtype, x.device)
        return layer(x, y, algo=algo, stream=stream)

    def _forward(self, x, algo, keep, stream):
        for spec in self.stem:
            x = self._conv(spec, x, algo, stream)
            if keep is not None:
                keep[spec.name] = x
        for blk in self.blocks:
            inp = x
            join = None
            if blk.shortcut is None:
                sc = inp
            elif stream is None:
                # the strided 1x1x1 projection is independent of the block's main path: side stream, joined
                # before the residual is added (a parallel branch when captured into a CUDA graph)
                if self.side is None:
                    self.side = torch.cuda.Stream(device=x.device)
                main = torch.cuda.current_stream(x.device)
                _wait(self.side, _record(main))
                with torch.cuda.stream(self.side), B.concurrent_kernels():
                    sc = self._conv(blk.shortcut, inp, algo, None)
                    join = _record(self.side)
            else:
                sc = self._conv(blk.shortcut, inp, algo, stream)
            # until the join, the main path's kernels run beside the projection on the side stream
            beside = B.concurrent_kernels() if join is not None else contextlib.nullcontext()
            beside.__enter__()
            if keep is not None and blk.shortcut is not None:
                keep[blk.shortcut.name] = sc
            last = blk.convs[-1]
            if self.fuse_pairs and keep is None and algo == B.ALGO_AUTO:
                c = blk.convs
                y = self._pair(c[0], c[1], x, None, c[1].relu, stream, c[1].name)
                x = y if y is not None else self._conv(c[1], self._conv(c[0], x, algo, stream), algo, stream)
                beside.__exit__(None, None, None)
                if join is not None:
                    _wait(torch.cuda.current_stream(x.device), join)
                y = self._pair(c[2], c[3], x, sc, True, stream, blk.name + ".out")
                if y is None:
                    x = self._conv(c[2], x, algo, stream)
                    layer = self.layers[last.name]
                    y = self.ws.get(blk.name + ".out", layer.out_shape(x), x.dtype, x.device)
                    y = layer.fused(x, y, residual=sc, relu=True, algo=algo, stream=stream)
                x = y
                continue
            for spec in blk.convs[:-1] if self.fuse_residual else blk.convs:
                x = self._conv(spec, x, algo, stream)
                if keep is not None:
                    keep[spec.name] = x
            beside.__exit__(None, None, None)
            if join is not None:
                _wait(torch.cuda.current_stream(x.device), join)
            if self.fuse_residual:
                layer = self.layers[last.name]
                y = self.ws.get(blk.name + ".out", layer.out_shape(x), x.dtype, x.device)
                x = layer.fused(x, y, residual=sc, relu=True, algo=algo, stream=stream)
            else:
                y = self.ws.get(blk.name + ".out", x.shape, x.dtype, x.device)
                x = add_relu(x, sc, last.cout, True, y, stream=stream)
            if keep is not None:
                keep[blk.name + ".out"] = x
        return x

    def n_launches(self) -> int:
        """Launches of one forward pass (after a first pass has found out which pairs the library fuses)."""
        per_block = 4 if self.fuse_residual else 5
        return len(self.stem) + sum(per_block + (blk.shortcut is not None) for blk in self.blocks) - len(self.pairs_fused)


class S3DNet(_NotedForward):
    """S3D-shaped forward (separable 3-D Inception): stem convs and pools, then Inception blocks whose four
    branches write straight into their channel slice of the block's output tensor (no concat pass)."""

    _SWITCHES = ("plan", "input_pad_zero", "parallel_branches", "ws")

    def _all_layers(self):
        return list(self.layers.values())

    def __init__(self, plan, layers, input_pad_zero: bool = True, parallel_branches: bool = True):
        self.plan, self.layers = plan, layers
        self.input_pad_zero = input_pad_zero
        # The four branches of an Inception block are independent and mostly too small to fill the GPU (a few
        # dozen tiles each): run them on separate streams, joined before the next block.  Inside a CUDA graph
        # capture this becomes parallel branches of the graph.  (Only with the default stream argument.)
        self.parallel_branches = parallel_branches
        self.side = None
        self.ws = Workspace()

    def _branch_streams(self, device):
        if self.side is None:
            self.side = [torch.cuda.Stream(device=device) for _ in range(3)]
        return self.side

    def _conv(self, spec, x, algo, stream, pad0=False):
        layer = self.layers[spec.name]
        y = self.ws.get(spec.name, layer.out_shape(x), x.dtype, x.device)
        return layer(x, y, algo=algo, stream=stream, x_pad_zero=pad0)

    def _concat(self, specs):
        """The layers of `specs`, which read the same tensor, as one; None where their handles do not go together."""
        parts = [self.layers[sp.name] for sp in specs]
        made = self.__dict__.setdefault("_concats", {})
        key = tuple(sp.name for sp in specs)
        now = [(p.packed, bool(p.packed.handle), p.spec, p.bias is None) for p in parts]
        if key not in made or made[key][0] != now:
            layer = None
            specs = [p.spec for p in parts]
            if all(sp.relu == specs[0].relu and sp.stride == specs[0].stride and sp.pad == specs[0].pad for sp in specs) and \
                    len({p.dtype for p in parts}) == 1 and all(sp.cout % 8 == 0 for sp in specs):
                try:
                    packed = B.rt3d_pack_concat([p.packed for p in parts])
                except B.Rt3dError as e:
                    if e.status != B.ERR_SHAPE:
                        raise
                else:
                    layer = object.__new__(ConvLayer)
                    cout = sum(sp.cout for sp in specs)
                    vars(layer).update(             # no assignment: what other passes have noted still holds
                        spec=dataclasses.replace(specs[0], name="+".join(key), cout=cout), packed=packed, _params={},
                        dtype=parts[0].dtype, dense=parts[0].dense, device=parts[0].device,
                        # filled from the parts' biases by _merged at every pass
                        bias=torch.empty(cout, device=parts[0].device) if any(p.bias is not None for p in parts) else None)
            made[key] = (now, layer)
        return made[key][1]

    def _merged(self, stream):
        """The merged convolutions by block name: (all three, None), (None, the two reductions) or neither.  Their biases are
        brought together in one launch on the device: every pass, a captured one too, reads what the layers' biases hold."""
        found, copies = {}, []
        for i, op in enumerate(self.plan):
            if not hasattr(op, "b0"):
                continue
            last = i + 1 == len(self.plan)
            specs = (op.b1[0], op.b2[0]) if last else (op.b1[0], op.b2[0], op.b0)
            layer = self._concat(specs)
            found[op.name] = (None, layer) if last else (layer, None)
            if layer is not None and layer.bias is not None:
                first = 0
                for part in (self.layers[sp.name] for sp in specs):
                    copies.append((part.bias, layer.bias, first, part.spec.cout))
                    first += part.spec.cout
        if copies:
            B.rt3d_copy_f32(copies, stream)
        return found

    def _block(self, op, x, off, algo, stream, merged):
        """One Inception block on channels [off, off + cin) of x; returns (output tensor, first channel of the output in it).

        The three 1x1x1 convolutions that read the block's input run as one where the layers allow it (`merged`): a third of
        the reads of x and of the launches.  It writes [b1 reduction | b2 reduction | b0] side by side, so the block's output
        then lies behind the reductions in one wide tensor, on a 128-byte boundary; the last block, whose output is the
        network's, merges the two reductions only."""
        n, t, h, w, _ = x.shape
        xd = B.channel_slice_desc(x, off, op.cin)
        r1, r2 = op.b1[0].cout, op.b2[0].cout
        wide, both = merged
        if wide is not None:
            start = -(-(r1 + r2) // 64) * 64                        # first channel of the output
            out = self.ws.get(op.name + ".wide", (n, t, h, w, start + -(-op.cout // 64) * 64), x.dtype, x.device)
            red, red_off = out, start - r1 - r2
        else:
            start, red_off = 0, 0
            out = self.ws.get(op.name, (n, t, h, w, op.cout), x.dtype, x.device)
            red = None if both is None else self.ws.get(op.name + ".reduce", (n, t, h, w, r1 + r2), x.dtype, x.device)
        offs = [start, start + op.b0.cout, start + op.b0.cout + op.b1[2].cout, start + op.b0.cout + op.b1[2].cout + op.b2[2].cout]

        def branch0():
            self.layers[op.b0.name].run_desc(xd, B.channel_slice_desc(out, offs[0], op.b0.cout), algo, stream)

        def sep(br, to, at):
            if red is None:
                a = self.ws.get(br[0].name, self.layers[br[0].name].out_shape(x), x.dtype, x.device)
                ad = B.tensor_desc(a, br[0].cout)
                self.layers[br[0].name].run_desc(xd, ad, algo, stream)
            else:
                ad = B.channel_slice_desc(red, at, br[0].cout)
            b = self.ws.get(br[1].name, (n, t, h, w, pitch_for(br[1].cout, x.dtype)), x.dtype, x.device)
            self.layers[br[1].name].run_desc(ad, B.tensor_desc(b, br[1].cout), algo, stream)
            self.layers[br[2].name].run_desc(B.tensor_desc(b, br[2].cin), B.channel_slice_desc(out, to, br[2].cout), algo, stream)

        def branch3():
            p = self.ws.get(op.pool.name, (n, t, h, w, pitch_for(op.cin, x.dtype)), x.dtype, x.device)
            B.rt3d_maxpool3d(xd, op.pool.k, op.pool.stride, op.pool.pad, B.tensor_desc(p, op.cin), stream)
            self.layers[op.b3.name].run_desc(B.tensor_desc(p, op.cin), B.channel_slice_desc(out, offs[3], op.b3.cout), algo, stream)

        def reduce():
            layer = wide if wide is not None else both
            if layer is not None:
                layer.run_desc(xd, B.channel_slice_desc(red, red_off, layer.spec.cout), algo, stream)

        seps = [lambda: sep(op.b1, offs[1], red_off), lambda: sep(op.b2, offs[2], red_off + r1)]
        rest = branch0 if wide is None else None
        if not (self.parallel_branches and stream is None):
            reduce()
            for fn in ([rest] if rest else []) + seps + [branch3]:
                fn()
            return out, start
        # independent branches on streams of their own; the main stream takes the reductions and the longest branch
        main, side = torch.cuda.current_stream(x.device), self._branch_streams(x.device)
        joins = []
        with B.concurrent_kernels():
            def beside(s, fn, after):
                _wait(s, after)
                with torch.cuda.stream(s):
                    fn()
                    joins.append(_record(s))

            fork = _record(main)
            beside(side[2], branch3, fork)
            if rest is not None:
                beside(side[0], rest, fork)
            reduce()
            beside(side[1], seps[1], _record(main) if red is not None else fork)
            seps[0]()
        for ev in joins:
            _wait(main, ev)
        return out, start

    def _forward(self, x, algo, keep, stream):
        c, off = self.plan[0].cin, 0
        merged = self._merged(stream) if keep is None else {}
        for i, op in enumerate(self.plan):
            if hasattr(op, "b0"):                                   # Inception block
                x, off = self._block(op, x, off, algo, stream, merged.get(op.name, (None, None)))
                c = op.cout
            elif hasattr(op, "cout"):
                if off:                                             # behind a wide block
                    y = self.ws.get(op.name, self.layers[op.name].out_shape(x), x.dtype, x.device)
                    self.layers[op.name].run_desc(B.channel_slice_desc(x, off, c), B.tensor_desc(y, op.cout), algo, stream)
                    x = y
                else:
                    x = self._conv(op, x, algo, stream, pad0=self.input_pad_zero and i == 0)
                c, off = op.cout, 0
            else:
                n, t, h, w, cs = x.shape
                ext = [(d + 2 * p - k) // s + 1 for d, p, k, s in zip((t, h, w), op.pad, op.k, op.stride)]
                y = self.ws.get(op.name, (n, ext[0], ext[1], ext[2], pitch_for(c, x.dtype)), x.dtype, x.device)
                B.rt3d_maxpool3d(B.channel_slice_desc(x, off, c), op.k, op.stride, op.pad, B.tensor_desc(y, c), stream)
                x, off = y, 0
            if keep is not None:
                keep[op.name] = x
        return x


class GraphedForward:
    """A network forward pass captured once into a CUDA graph and replayed: removes the host-side
    launch cost of the 13-45 kernels of a forward pass (at batch 1 the kernels are shorter than the
    launches).  The input buffer is fixed at capture time; copy new clips into `self.x` before replay."""

    def __init__(self, net, x: torch.Tensor, algo=B.ALGO_AUTO):
        self.net, self.x = net, x
        net.forward(x, algo=algo)                    # first use: weight upload, workspaces, function attributes
        net.forward(x, algo=algo)
        torch.cuda.synchronize()
        self.graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(self.graph):
            self.y = net.forward(self.x, algo=algo)

    def __call__(self) -> torch.Tensor:
        self.graph.replay()
        return self.y

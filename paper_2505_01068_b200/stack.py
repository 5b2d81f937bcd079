"""The GsiT fusion stack as a sequence of library calls (Eq. "All-Modal-In-One fusion"): a forward-ring
encoder and a backward-ring encoder, each with its own weights, both starting from the same input; their
outputs side by side on the feature axis (width 2d); then the intra-modal encoder on that.  Only
sequencing and buffer reuse happen here -- each layer is one gsit_im_layer_fwd call, and the feature
concat costs nothing because the last layer of each ring writes its half of the [B, L, 2d] buffer.

The two rings share nothing but their input: their layers of equal depth go through one library call each (one launch per
kernel for both).  All launches of such a forward are issued by one call of the extension (csrc/torch_ext.cpp).  Rings of
unequal depth, or paired_rings=False, are issued from Python on two CUDA streams (fork after the input is ready, join
before the intra encoder), each ring with its own workspace and ping-pong buffers."""
from __future__ import annotations

import torch

from . import binding as B


class GsitStack:
    def __init__(self, fwd_layers, bwd_layers, intra_layers, seg_len, heads, intra_heads, ln_eps=1e-5, head=None,
                 concurrent_rings=True, batch_chunks=1, intra_halves=True,
                 packed=True, paired_rings=True):
        """head: optional (w_f, b_f) of the read-out X_m = f(|| Split(.)[-1]); see read_out().
        packed: when valid lengths are given (and the layers are bf16 at widths 32, 64 or 128 with heads up to 32), the
        stack works on the packed row layout: the real rows are gathered once, every layer runs on them only, and the
        result is scattered back with +0 in the padded positions.  The row-wise parts of the layers then do no work
        for padding (24 % of the rows at the benchmark's lengths).  The plan of where each segment starts is made on the
        device, so a captured forward stays valid when the lengths change.
        paired_rings: (rings of equal depth) the forward-ring and backward-ring layers of equal depth go through one
        gsit_im_layer_pair_fwd call each, and the whole forward is issued on the caller's stream, each launch starting
        under the tail of the one before it.
        The other options belong to forwards whose rings are not paired (paired_rings=False, rings of unequal depth) or to
        batch_chunks > 1.  concurrent_rings: issue independent work on several streams (False: every launch on the caller's
        stream).  batch_chunks: the batch is cut into this many groups of samples, each with its own pair of streams;
        samples never interact, so it changes the result by rounding at most
        (where a group's size selects another attention kernel).  intra_halves: the intra encoder runs on the two
        halves of the batch on the two streams (in a captured graph within 1 % of the whole batch per launch at 2, 16 and 64
        samples of 1050 rows; issued call by call 276 against 232 us at 2, the same from 16 on)."""
        self.head = head
        self.concurrent_rings = concurrent_rings
        self.batch_chunks = max(1, int(batch_chunks))
        self.intra_halves = bool(intra_halves)
        self.packed = bool(packed)
        self.paired_rings = bool(paired_rings)
        self.fwd, self.bwd, self.intra = list(fwd_layers), list(bwd_layers), list(intra_layers)
        self.seg_len, self.heads, self.intra_heads, self.ln_eps = tuple(seg_len), heads, intra_heads, ln_eps
        self._bufs = None
        self._lanes = None  # streams and events of the concurrent issue, created on first use
        self._ring_done = None

    def _chunks(self, Bn):
        nch = min(self.batch_chunks, Bn) if (self.concurrent_rings and self.fwd and self.bwd) else 1
        q, r = divmod(Bn, nch)
        out, lo = [], 0
        for c in range(nch):
            hi = lo + q + (1 if c < r else 0)
            out.append(slice(lo, hi))
            lo = hi
        return out

    def _workspace_need(self, Bn, d, valid_len, plan=None, capacity=0):
        """Bytes that the most demanding layer of the stack asks for (layers may differ in type and MLP width)."""
        need = 0
        for layers, width, heads, phase in ((self.fwd + self.bwd, d, self.heads, B.PHASE_INTER_FWD), (self.intra, 2 * d, self.intra_heads, B.PHASE_INTRA)):
            for t, d_ff in {(w["w_qkv"].dtype, w["w_1"].shape[0]) for w in layers}:
                sh = B.make_shape(Bn, self.seg_len, width, heads, valid_len, B._dtype_code(t), phase, row_start=plan, capacity=capacity)
                need = max(need, B.workspace_bytes(sh, B.CALL_LAYER, d_ff))
        return need

    def _buffers(self, x, valid_len):
        Bn, L, d = x.shape
        chunks = self._chunks(Bn)
        key = (Bn, L, d, x.device, len(chunks))
        if self._bufs is None:
            self._bufs = {}
        if key not in self._bufs:
            ws = []
            for sl in chunks:  # two workspaces per chunk of the batch: one per ring (the intra encoder reuses the first)
                need = self._workspace_need(sl.stop - sl.start, d, None if valid_len is None else valid_len[sl])
                ws.append([torch.empty(need, dtype=torch.uint8, device=x.device) for _ in range(2)])
            f32 = dict(dtype=torch.float32, device=x.device)
            self._bufs[key] = (ws, [torch.empty((Bn, L, d), **f32) for _ in range(4)],
                               torch.empty((Bn, L, 2 * d), **f32), torch.empty((Bn, L, 2 * d), **f32))
        return (chunks,) + self._bufs[key]

    def _ring(self, x, layers, phase, half, c0, ws, ping, valid_len):
        d = x.shape[2]
        cur = x
        for i, w in enumerate(layers):
            dst = c0[:, :, half * d:(half + 1) * d] if i == len(layers) - 1 else ping[i % 2]
            B.im_layer_fwd(cur, w, self.seg_len, self.heads, valid_len, phase, ln_eps=self.ln_eps, out=dst, workspace=ws)
            cur = dst

    def _intra(self, c0, c1, ws, valid_len):
        cur, ping = c0, [c1, c0]
        for i, w in enumerate(self.intra):
            dst = ping[i % 2]
            B.im_layer_fwd(cur, w, self.seg_len, self.intra_heads, valid_len, B.PHASE_INTRA, ln_eps=self.ln_eps,
                           out=dst, workspace=ws)
            cur = dst
        return len(self.intra) % 2  # 1: the result is in c1, 0: in c0

    def _packed_buffers(self, x, valid_len):
        Bn, L, d = x.shape
        key = ("packed", Bn, L, d, x.device)
        if self._bufs is None:
            self._bufs = {}
        if key not in self._bufs:
            cap = Bn * L + 128  # always enough: the real rows plus the alignment of the second half's first row
            plan = torch.zeros(3 * Bn + 1, dtype=torch.int32, device=x.device)
            need = self._workspace_need(Bn, d, valid_len, plan, cap)
            f32 = dict(dtype=torch.float32, device=x.device)
            ws_all = torch.empty(2 * need, dtype=torch.uint8, device=x.device)   # one per ring
            self._bufs[key] = (cap, plan, [ws_all[:need], ws_all[need:]],
                               [torch.zeros((cap, d), **f32) for _ in range(5)],
                               torch.zeros((cap, 2 * d), **f32), torch.zeros((cap, 2 * d), **f32),
                               torch.empty((Bn, L, 2 * d), **f32))
        return self._bufs[key]

    def _forward_packed(self, x, valid_len, out=None):
        cap, plan, ws, t, c0, c1, y = self._packed_buffers(x, valid_len)
        if out is not None:
            y = out
        Bn, L, d = x.shape
        conc = self.concurrent_rings and self.fwd and self.bwd
        halves = conc and self.intra_halves and self.intra and Bn >= 2
        mid = Bn // 2
        B.plan_rows(valid_len, self.seg_len, mid if halves else 0, out=plan)
        xp = B.pack_rows(x, t[4], self.seg_len, valid_len, plan)

        def ring(layers, phase, half, w_s, ping):
            cur = xp
            for i, w in enumerate(layers):
                dst = c0[:, half * d:(half + 1) * d] if i == len(layers) - 1 else ping[i % 2]
                B.im_layer_fwd(cur, w, self.seg_len, self.heads, valid_len, phase, ln_eps=self.ln_eps, out=dst, workspace=w_s,
                               row_start=plan)
                cur = dst

        def intra(lo, hi, w_s):  # samples lo .. hi - 1: their rows of the packed matrices are addressed through the plan
            cur, ping = c0, [c1, c0]
            for i, w in enumerate(self.intra):
                dst = ping[i % 2]
                B.im_layer_fwd(cur, w, self.seg_len, self.intra_heads, valid_len[lo:hi], B.PHASE_INTRA, ln_eps=self.ln_eps,
                               out=dst, workspace=w_s, row_start=plan[3 * lo:])
                cur = dst
            return cur

        if not conc:
            ring(self.fwd, B.PHASE_INTER_FWD, 0, ws[0], t[0:2])
            ring(self.bwd, B.PHASE_INTER_BWD, 1, ws[0], t[0:2])
            res = intra(0, Bn, ws[0]) if self.intra else c0
        else:
            if self._lanes is None:
                dev = x.device
                self._lanes = ([torch.cuda.Stream(device=dev) for _ in range(2)], torch.cuda.Event(),
                               [torch.cuda.Event() for _ in range(2)])
                self._ring_done = [torch.cuda.Event()]
            streams, fork, done = self._lanes
            s_f, s_b = streams[0], streams[1]
            main = torch.cuda.current_stream(x.device)
            fork.record(main)
            s_f.wait_event(fork)
            s_b.wait_event(fork)
            with torch.cuda.stream(s_b):
                ring(self.bwd, B.PHASE_INTER_BWD, 1, ws[1], t[2:4])
                done[1].record(s_b)
            with torch.cuda.stream(s_f):
                ring(self.fwd, B.PHASE_INTER_FWD, 0, ws[0], t[0:2])
                res = c0
                if halves:
                    ring_f = self._ring_done[0]
                    ring_f.record(s_f)
                    s_f.wait_event(done[1])
                    res = intra(0, mid, ws[0])
                    with torch.cuda.stream(s_b):
                        s_b.wait_event(ring_f)
                        intra(mid, Bn, ws[1])
                        done[1].record(s_b)
                    s_f.wait_event(done[1])
                else:
                    s_f.wait_event(done[1])
                    if self.intra:
                        res = intra(0, Bn, ws[0])
                done[0].record(s_f)
            main.wait_event(done[0])
            for st in streams:
                x.record_stream(st)
                valid_len.record_stream(st)
        B.unpack_rows(res, y, self.seg_len, valid_len, plan)
        return y

    def forward(self, x, valid_len=None, out=None, check=False):
        """x float32 [B, L, d] -> float32 [B, L, 2d].  The result lives in a buffer owned by this object, or in `out`
        (float32 [B, L, 2d], contiguous) when one is given.  x may lie anywhere in `out`, and with paired rings or packed rows also in
        the owned buffer (a view of the result before), which then no longer holds it afterwards.  check=True synchronises the stream afterwards and raises
        GsitError if a kernel reported a timed-out device-side wait (not for use under stream capture)."""
        if out is not None:
            assert out.shape == (x.shape[0], x.shape[1], 2 * x.shape[2]) and out.dtype == torch.float32 and out.is_contiguous()
        res = self._forward(x, valid_len, out)
        if out is not None and res.data_ptr() != out.data_ptr():
            out.copy_(res)
            res = out
        if check:
            code, flags = B.last_device_status()
            if code != 0:
                raise B.GsitError(code, f"GsitStack.forward: device status flags {flags:#x}")
        return res

    def _native_buffers(self, x, valid_len, packed):
        """Buffers of the natively issued forward, kept per problem size: (the ten tensors stack_forward takes, result)."""
        key = ("native", packed, x.shape, x.device)
        got = None if self._bufs is None else self._bufs.get(key)
        if got is not None:
            return got
        Bn, L, d = x.shape
        cap = Bn * L + 128 if packed else Bn * L
        plan = torch.zeros(3 * Bn + 1, dtype=torch.int32, device=x.device) if packed else None
        need = self._workspace_need(Bn, d, valid_len, plan, cap if packed else 0)
        # rows past the last real one are read by the last row tile (and discarded): they start out as zeros
        z = lambda cols: torch.zeros((cap, cols), dtype=torch.float32, device=x.device)
        bufs = (plan, torch.empty(2 * need, dtype=torch.uint8, device=x.device), z(d), z(d), z(d), z(d), z(d) if packed else None,
                z(2 * d), z(2 * d), torch.empty(cap, dtype=torch.int32, device=x.device) if packed else None)
        if self._bufs is None:
            self._bufs = {}
        got = self._bufs[key] = (bufs, torch.empty((Bn, L, 2 * d), dtype=torch.float32, device=x.device))
        return got

    def _forward_native(self, x, valid_len, out):
        """One call that issues every launch of the forward (about 2 us each; issuing them from Python took 15)."""
        packed = self.packed and valid_len is not None
        while True:
            bufs, y = self._native_buffers(x, valid_len, packed)
            if out is not None:
                y = out
            code = B.native().stack_forward(x, valid_len, y, self.fwd, self.bwd, self.intra, self.seg_len, self.heads, self.intra_heads,
                                            self.ln_eps, bufs)
            if code == 0:
                return y
            if not (packed and code == 2):  # anything but "this shape is not covered in the packed layout": a real error
                raise B.GsitError(code, "GsitStack.forward")
            packed = self.packed = False

    def _forward(self, x, valid_len, out):
        if self.paired_rings and self.batch_chunks == 1 and len(self.fwd) == len(self.bwd) > 0:
            return self._forward_native(x, valid_len, out)
        if self.packed and valid_len is not None and self.batch_chunks == 1:
            try:
                return self._forward_packed(x, valid_len, out)
            except B.GsitError as e:
                if e.code != 2:  # anything but "this shape is not covered": a real error
                    raise
                self.packed = False
        chunks, ws, t, c0, c1 = self._buffers(x, valid_len)
        if len(chunks) == 1 and not (self.concurrent_rings and self.fwd and self.bwd):
            self._ring(x, self.fwd, B.PHASE_INTER_FWD, 0, c0, ws[0][0], t[0:2], valid_len)
            self._ring(x, self.bwd, B.PHASE_INTER_BWD, 1, c0, ws[0][0], t[0:2], valid_len)
            return c1 if self._intra(c0, c1, ws[0][0], valid_len) else c0
        nch = len(chunks)
        if self._lanes is None or len(self._lanes[0]) != 2 * nch:
            dev = x.device
            self._lanes = ([torch.cuda.Stream(device=dev) for _ in range(2 * nch)], torch.cuda.Event(),
                           [torch.cuda.Event() for _ in range(2 * nch)])
            self._ring_done = [torch.cuda.Event() for _ in range(nch)]
        streams, fork, done = self._lanes
        main = torch.cuda.current_stream(x.device)
        fork.record(main)
        for c, sl in enumerate(chunks):
            vl = None if valid_len is None else valid_len[sl]
            s_f, s_b = streams[2 * c], streams[2 * c + 1]
            s_f.wait_event(fork)
            s_b.wait_event(fork)
            with torch.cuda.stream(s_b):
                self._ring(x[sl], self.bwd, B.PHASE_INTER_BWD, 1, c0[sl], ws[c][1], [t[2][sl], t[3][sl]], vl)
                done[2 * c + 1].record(s_b)
            with torch.cuda.stream(s_f):
                self._ring(x[sl], self.fwd, B.PHASE_INTER_FWD, 0, c0[sl], ws[c][0], [t[0][sl], t[1][sl]], vl)
                n = sl.stop - sl.start
                if self.intra_halves and self.intra and n >= 2:
                    # both streams wait for both rings, then each runs the intra encoder on one half of the samples
                    # (the ring workspaces are free by then: one per half)
                    lo, hi = slice(sl.start, sl.start + n // 2), slice(sl.start + n // 2, sl.stop)
                    ring_f = self._ring_done[c]
                    ring_f.record(s_f)
                    s_f.wait_event(done[2 * c + 1])
                    which = self._intra(c0[lo], c1[lo], ws[c][0], None if valid_len is None else valid_len[lo])
                    with torch.cuda.stream(s_b):
                        s_b.wait_event(ring_f)
                        self._intra(c0[hi], c1[hi], ws[c][1], None if valid_len is None else valid_len[hi])
                        done[2 * c + 1].record(s_b)
                    s_f.wait_event(done[2 * c + 1])
                else:
                    s_f.wait_event(done[2 * c + 1])  # both rings of this chunk are complete
                    which = self._intra(c0[sl], c1[sl], ws[c][0], vl)
                done[2 * c].record(s_f)
        for c in range(nch):
            main.wait_event(done[2 * c])
        for st in streams:
            x.record_stream(st)
            if valid_len is not None:
                valid_len.record_stream(st)
        return c1 if which else c0

    def read_out(self, c, valid_len=None):
        """X_m = f(|| Split(c)[-1]): last real step of each modality of the stack output c [B, L, 2d], through the linear
        map given as `head` -> float32 [B, out_features] (one gsit_stack_head_fwd call)."""
        assert self.head is not None, "no read-out weights were given"
        w_f, b_f = self.head
        return B.stack_head_fwd(c, w_f, b_f, self.seg_len, valid_len)

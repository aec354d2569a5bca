"""Buffer management around the two library calls (PyTorch is used for device memory and streams only)."""

import threading
import weakref

import torch

from . import binding as B


class _Uploads:
    """The stream on which the host-buffer calls made on one stream copy their inputs, whichever layers they are for.  Their
    copies are then served in the order of the calls; with a stream per layer the copy engine shared itself out between the
    inputs of this call and those of calls several places behind it (three layers in rotation, 100 frames: 28.0 ms a call instead of
    24).  Calls on one stream follow one another there in any case.  Those of another stream have copies of their own,
    which wait for nothing of this one's."""

    def __init__(self, index):
        self.stream = torch.cuda.Stream(index)

    _of_caller = weakref.WeakValueDictionary()   # (device index, caller's stream) -> _Uploads; kept by the layers that use it
    _lock = threading.Lock()

    @classmethod
    def of(cls, index, caller):
        with cls._lock:
            uploads = cls._of_caller.get((index, caller.cuda_stream))
            if uploads is None:
                uploads = cls._of_caller[index, caller.cuda_stream] = cls(index)
            return uploads


def host_groups(n_frames, n_chunks):
    """Boundaries of ``n_chunks`` groups of frames, none empty: equal ones, but with small groups at both ends, since the
    attention of a call begins after the copy of the first group's Q and the call ends with the copy of the last
    group's output."""
    weights = [1.0] * n_chunks
    if n_chunks > 4:
        weights[:2], weights[-2:] = [0.25, 0.5], [0.5, 0.25]
    bounds, total, seen = [0], sum(weights), 0.0
    for i, w in enumerate(weights):
        seen += w
        bounds.append(min(max(round(seen / total * n_frames), bounds[-1] + 1), n_frames - (n_chunks - 1 - i)))
    return bounds


class SubsampledGlobalAttention:
    """Owns the compact K/V, the mean pair, the index list and the workspaces of one problem shape
    and runs the two C-ABI calls on the current CUDA stream.

    ``forward(Q, K, V)`` takes bf16 CUDA tensors [N*L, H, d] and returns O of the same shape.
    """

    def __init__(self, params, device="cuda", want_lse=False):
        if not torch.cuda.is_available():
            raise RuntimeError("libavggt needs a CUDA device (sm_100); there is no CPU fallback")
        self.params = params
        self.device = torch.device(device)
        self._index = torch.cuda.current_device() if self.device.index is None else self.device.index
        with torch.cuda.device(self.device):
            self.M, self.n_dropped = B.avggt_kv_count(params)
            self.build_ws_bytes, self.attn_ws_bytes = B.avggt_workspace_bytes(params)
        H, d = params.n_heads, params.head_dim
        self.n_tok = params.n_frames * params.tokens_per_frame
        self._shape = torch.Size((self.n_tok, H, d))
        dev = self.device
        self.Kc = torch.empty((H, self.M, d), dtype=torch.bfloat16, device=dev)
        self.Vc = torch.empty((H, self.M, d), dtype=torch.bfloat16, device=dev)
        self.idx = torch.empty((self.M,), dtype=torch.int32, device=dev)
        self.kmean = torch.zeros((H, d), dtype=torch.float32, device=dev)
        self.vmean = torch.zeros((H, d), dtype=torch.float32, device=dev)
        self.build_ws = torch.empty((max(self.build_ws_bytes, 16),), dtype=torch.uint8, device=dev)
        self.attn_ws = torch.zeros((max(self.attn_ws_bytes, 16),), dtype=torch.uint8, device=dev)
        self.lse = torch.empty((self.n_tok, H), dtype=torch.float32, device=dev) if want_lse else None

    def _stream(self):
        # what torch.cuda.current_stream(device).cuda_stream gives, without building the Stream object (4 us of a 30 us layer)
        return torch._C._cuda_getCurrentRawStream(self._index)

    def build_kv(self, K, V):
        B.avggt_build_kv(self.params, K, V, self.Kc, self.Vc, self.idx, self.kmean, self.vmean,
                         self.build_ws, self.build_ws.numel(), self._stream())

    def attend(self, Q, K, V, out=None):
        if out is None:
            out = torch.empty_like(Q)
        B.avggt_global_attn(self.params, Q, K, V, self.Kc, self.Vc, self.kmean, self.vmean, out, self.lse,
                            self.attn_ws, self.attn_ws.numel(), self._stream())
        return out

    def frame_attend(self, Q, K, V, out=None):
        """Frame attention (a converted early global block): each frame attends to itself only."""
        self._check_inputs(Q, K, V)
        if out is None:
            out = torch.empty_like(Q)
        with torch.cuda.device(self._index):
            B.avggt_frame_attn(self.params, Q, K, V, out, self.lse, self.attn_ws, self.attn_ws.numel(), self._stream())
        return out

    def forward(self, Q, K, V, out=None):
        self._check_inputs(Q, K, V)
        if torch.cuda.current_device() != self._index:
            with torch.cuda.device(self._index):
                return self._layer(Q, K, V, out)
        return self._layer(Q, K, V, out)

    __call__ = forward

    def _layer(self, Q, K, V, out):
        if out is None:
            out = torch.empty_like(Q)
        B.avggt_layer(self.params, Q, K, V, self.Kc, self.Vc, self.idx, self.kmean, self.vmean, out, self.lse, self.build_ws,
                      self.build_ws.numel(), self.attn_ws, self.attn_ws.numel(), self._stream())
        return out

    def forward_host(self, hQ, hK, hV, hO, n_chunks=8, inputs_ready=None):
        """The layer on host buffers (pinned memory), with the copies hidden behind the kernels.

        K and V go to the device first (the compaction and the mean need all of them); Q then arrives in
        ``n_chunks`` groups of frames on a copy stream while the attention of the previous group runs
        (``avggt_global_attn_shard``: the queries of a frame range against the whole sequence's compact keys), and
        every group's output leaves on a second copy stream.  The groups' kernels take turns on the current stream and a
        stream of the layer's own, so that the thread blocks of a group move in as those of the group before run out
        (eight launches in a row on one stream left a tenth of the chip's time unused: 100 frames 28.0 -> 27.2 ms a call,
        33.3 -> 30.7 ms for a call on its own).  The call returns without waiting for the device: what it does is ordered
        with events, and the current stream waits for the last output copy.

        The inputs must be in the host buffers when the call is made: their copies do not wait for the current stream, which
        is what lets them travel under the call before.  Where something on the device still writes them (an asynchronous copy to the
        host), pass the event recorded behind it as ``inputs_ready``.  ``hO`` is written after what is on the current stream.

        The device copies of K and V alternate between two buffers, so that the K and V of a call made right after this one
        travel while this one's attention runs; Q and O have one buffer, guarded group by group.  The device
        staging buffers are allocated on first use.
        """
        p = self.params
        dev = self.device
        cur = torch.cuda.current_stream(dev)
        if not hasattr(self, "_host_path"):
            shape = (self.n_tok, p.n_heads, p.head_dim)
            new = lambda: torch.empty(shape, dtype=torch.bfloat16, device=dev)
            self._host_path = dict(
                Q=new(), O=new(), K=[new(), new()], V=[new(), new()], uploads=None, d2h=torch.cuda.Stream(dev),
                turn=torch.cuda.Stream(dev),
                calls=0,
                uploaded=None,           # the previous call's inputs have arrived
                kv_free=[[], []],        # per K/V buffer: the call that used it last has finished with it
                bounds=None,             # frame groups of the previous call
                q_free=[], o_free=[],    # per group of the previous call: its attention has read Q / its output copy has left O
                # one status block per group of frames, so that no launch clears what an earlier one reported
                ws=torch.zeros((max(1, p.n_frames), max(self.attn_ws_bytes, 256)), dtype=torch.uint8, device=dev))
        hp = self._host_path
        which = hp["calls"] & 1
        hp["calls"] += 1
        dQ, dK, dV, dO, d2h = hp["Q"], hp["K"][which], hp["V"][which], hp["O"], hp["d2h"]
        hp["uploads"] = _Uploads.of(self._index, cur)
        h2d = hp["uploads"].stream
        if hp["uploaded"] is not None:
            h2d.wait_event(hp["uploaded"])     # on another stream, perhaps
        L = p.tokens_per_frame
        n_chunks = max(1, min(n_chunks, p.n_frames))
        bounds = host_groups(p.n_frames, n_chunks)
        same_groups = hp["bounds"] == bounds
        keep_first = bool(p.flags & B.AVGGT_FLAG_KEEP_FIRST_FRAME)
        if not same_groups:
            # the previous call cut the frames differently: wait for all of it before Q and O are touched
            h2d.wait_stream(cur)
            h2d.wait_stream(d2h)
        with torch.cuda.device(dev):
            with torch.cuda.stream(h2d):
                if inputs_ready is not None:
                    h2d.wait_event(inputs_ready)
                for ev in hp["kv_free"][which]:
                    h2d.wait_event(ev)
                dK.copy_(hK, non_blocking=True)
                dV.copy_(hV, non_blocking=True)
                kv_ready = torch.cuda.Event()
                kv_ready.record(h2d)
                q_ready = []
                for c in range(n_chunks):
                    sl = slice(bounds[c] * L, bounds[c + 1] * L)
                    if same_groups:
                        h2d.wait_event(hp["q_free"][c])
                    dQ[sl].copy_(hQ[sl], non_blocking=True)
                    ev = torch.cuda.Event()
                    ev.record(h2d)
                    q_ready.append(ev)
            hp["uploaded"] = q_ready[-1]
            cur.wait_event(kv_ready)
            self.build_kv(dK, dV)
            built = torch.cuda.Event()
            built.record(cur)
            hp["turn"].wait_event(built)
            q_free, o_free = [], []
            for c in range(n_chunks):
                f0, f1 = bounds[c], bounds[c + 1]
                sl = slice(f0 * L, f1 * L)
                cp = B.make_params(f1 - f0, p.grid_h, p.grid_w, p.n_special, p.n_heads, p.head_dim, p.sigma, diag=p.diag,
                                   mean_fill=p.mean_fill, softmax_scale=p.softmax_scale,
                                   keep_first_frame=keep_first and f0 == 0)
                on = hp["turn"] if c & 1 else cur
                on.wait_event(q_ready[c])
                if same_groups:
                    on.wait_event(hp["o_free"][c])
                B.avggt_global_attn_shard(cp, self.M, self.n_dropped, dQ[sl], dK[sl], dV[sl], self.Kc, self.Vc, self.kmean,
                                          self.vmean, dO[sl], None, hp["ws"][c], hp["ws"][c].numel(), on.cuda_stream)
                done = torch.cuda.Event()
                done.record(on)
                q_free.append(done)
                d2h.wait_event(done)
                with torch.cuda.stream(d2h):
                    hO[sl].copy_(dO[sl], non_blocking=True)
                    left = torch.cuda.Event()
                    left.record(d2h)
                    o_free.append(left)
            hp["kv_free"][which] = q_free[-2:]     # the last group of either stream
            hp["bounds"], hp["q_free"], hp["o_free"] = bounds, q_free, o_free
            cur.wait_stream(d2h)
        return hO

    def check_status(self):
        """Synchronises the device and raises if a device-side wait gave up."""
        torch.cuda.synchronize(self.device)
        B.avggt_check_status(self.attn_ws)
        if hasattr(self, "_host_path"):
            for ws in self._host_path["ws"]:
                B.avggt_check_status(ws)

    def _check_inputs(self, *tensors):
        for t in tensors:
            if t.dtype is not torch.bfloat16 or t.shape != self._shape or not t.is_contiguous() or not t.is_cuda:
                raise ValueError(f"expected contiguous bf16 CUDA tensors of shape {tuple(self._shape)}")

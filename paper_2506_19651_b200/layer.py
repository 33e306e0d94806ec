"""One pass of the whole hot path over one layer's tensors, as a user of the library calls it.

Host-side orchestration only (buffer allocation through torch, then the C-ABI calls).  A pass is one call
(pevlm_layer_forward); its steps, in the order of the method, are RoPE at global positions with K and V written to the
caches -> parallel prefill attention (Eq. 3-4) and question attention (Eq. 5).
"""
from __future__ import annotations

from . import binding as pb


def _workspace(alloc, n_bytes):
    """A workspace whose status header (its first 256 bytes) reads as clear before the first call; the rest needs no value."""
    import torch
    ws = alloc((n_bytes,), torch.uint8)
    ws[:256].zero_()
    return ws


def _one_sequence(shape):
    if shape.batch != 1:
        raise ValueError(f"a layer pass is over one sequence, not a batch of {shape.batch}: its buffers hold the rows of one")


class LayerBuffers:
    """Device buffers of one layer pass over one sequence, allocated once and reused across steps."""

    def __init__(self, shape: pb.Shape, device="cuda", alloc=None):
        """`alloc(shape, dtype, zero)` replaces torch.empty / torch.zeros (the tests pass an allocator that puts
        guard bytes around every buffer)."""
        import torch
        s = shape
        _one_sequence(s)
        nv, Q, L = s.n_video, s.query_len, s.L
        Hq, Hkv, d = s.num_q_heads, s.num_kv_heads, s.head_dim
        bf, f32 = torch.bfloat16, torch.float32
        if alloc is None:
            def alloc(shp, dtype, zero=False):
                return (torch.zeros if zero else torch.empty)(shp, dtype=dtype, device=device)
        self.shape = s
        self.q_video = alloc((max(nv, 1), Hq, d), bf)   # roped copy of the video queries
        self.q_question = alloc((max(Q, 1), Hq, d), bf)
        self.k_cache = alloc((L, Hkv, d), bf)
        self.v_cache = alloc((L, Hkv, d), bf)
        self.o_video = alloc((max(nv, 1), Hq, d), bf)
        self.lse_video = alloc((Hq, max(nv, 1)), f32)
        self.o_question = alloc((max(Q, 1), Hq, d), bf)
        self.lse_question = alloc((Hq, max(Q, 1)), f32)
        self.ws_prefill = _workspace(alloc, pb.pevlm_workspace_bytes(s, pb.WS_PREFILL))
        self.ws_query = _workspace(alloc, pb.pevlm_workspace_bytes(s, pb.WS_QUERY))


def layer_forward(buf: LayerBuffers, q, k, v, mark=None):
    """q [L,Hq,d], k, v [L,Hkv,d]: un-roped bf16 device tensors of the whole stream.
    Leaves O/LSE of the video rows and of the question rows in `buf`.  `mark(name)`, if
    given, is called before the first call and after each C-ABI call (for event timing); without it the pass is one
    call (pevlm_layer_forward)."""
    s = buf.shape
    nv, Q = s.n_video, s.query_len
    _one_sequence(s)
    if mark is None:
        if nv + Q == 0:  # an empty stream is no call's shape
            return buf
        pb.pevlm_layer_forward(s, q, k, v, buf.q_video, buf.q_question, buf.k_cache, buf.v_cache, buf.o_video,
                               buf.lse_video, buf.o_question, buf.lse_question, buf.ws_prefill, buf.ws_query)
        return buf
    mark("start")
    if nv > 0:
        # K goes straight into its cache slot; Q is roped into a scratch copy
        pb.pevlm_rope_qk(s, q[:nv], k[:nv], buf.q_video, buf.k_cache[:nv], 0, nv)
        mark("rope_video")
        pb.pevlm_assemble_kv(s, None, v[:nv], None, None, buf.k_cache, buf.v_cache)
        mark("assemble_video")
        pb.pevlm_parallel_prefill_attn(s, buf.q_video, buf.k_cache[:nv], buf.v_cache[:nv], buf.o_video,
                                       buf.lse_video, buf.ws_prefill)
        mark("prefill_attn")
    if Q > 0:
        pb.pevlm_rope_qk(s, q[nv:], k[nv:], buf.q_question, buf.k_cache[nv:], nv, Q)
        mark("rope_question")
        pb.pevlm_assemble_kv(s, None, None, None, v[nv:], buf.k_cache, buf.v_cache)
        mark("assemble_question")
        pb.pevlm_query_attn(s, buf.q_question, buf.k_cache, buf.v_cache, buf.o_question, buf.lse_question,
                            buf.ws_query)
        mark("query_attn")
    return buf


def ragged_layer_forward(q, k, v, S, B, N, B_last, Q, theta, scale=0.0, alloc=None):
    """Layer pass over a video whose length is not a multiple of the block length: N context blocks, the
    first N-1 of B tokens, the last one of B_last < B tokens (the uniform partition of Sec. 3.2.1 with the
    remainder as one shorter block).  q [L,Hq,d], k, v [L,Hkv,d] un-roped device tensors of the whole
    stream, L = S + (N-1)*B + B_last + Q.  Returns (o_video, lse_video, o_question, lse_question, workspaces), the workspaces
    (for pevlm_read_status) being those of sink and full blocks, of the last block and of the question; the first two are one.

    One call (pevlm_layer_forward with the length of the last block); positions are the global ones.
    `alloc(shape, dtype, zero)` replaces torch.empty / torch.zeros (see LayerBuffers).
    """
    import torch
    Hq, Hkv, d = q.shape[1], k.shape[1], q.shape[2]
    nv = S + (N - 1) * B + B_last
    L = nv + Q
    assert N >= 1 and 1 <= B_last <= B and q.shape[0] == L
    bf, f32 = torch.bfloat16, torch.float32
    s = pb.make_shape(S, B, N, Q, Hq, Hkv, d, theta=theta, scale=scale)
    if alloc is None:
        # (new_empty takes type and device from the tensor: half of torch.empty's time on the host)
        def alloc(shp, dtype, zero=False):
            return q.new_empty(shp) if dtype is q.dtype else q.new_empty(shp, dtype=dtype)
    q_roped = alloc((L, Hq, d), bf)
    k_cache = alloc((L, Hkv, d), bf)
    v_cache = alloc((L, Hkv, d), bf)
    o_video = alloc((nv, Hq, d), bf)
    lse_video = alloc((Hq, nv), f32)
    o_question = alloc((max(Q, 1), Hq, d), bf)
    lse_question = alloc((Hq, max(Q, 1)), f32)
    # the launch writes the status words; a question that is not there leaves its own as it was
    ws_prefill = alloc((pb.pevlm_workspace_bytes(s, pb.WS_PREFILL),), torch.uint8)
    ws_query = (alloc((pb.pevlm_workspace_bytes(s, pb.WS_QUERY),), torch.uint8) if Q > 0
                else _workspace(alloc, pb.pevlm_workspace_bytes(s, pb.WS_QUERY)))
    pb.pevlm_layer_forward(s, q, k, v, q_roped, q_roped[nv:], k_cache, v_cache, o_video, lse_video, o_question, lse_question,
                           ws_prefill, ws_query, last_len=B_last)
    return o_video, lse_video, o_question, lse_question, [ws_prefill, ws_prefill, ws_query]


def _need_rows(n, q, k, v):
    """The calls get addresses only: that there are n rows behind them is seen to here."""
    if q.shape[0] < n or k.shape[0] < n or v.shape[0] < n:
        raise ValueError(f"{q.shape[0]}, {k.shape[0]}, {v.shape[0]} rows of q, k, v where {n} are read")


class StreamingWindow:
    """A sliding window of W context blocks over a fixed sink (the streaming use the paper names as
    future work, Sec. 5).  The cache is [sink | W block slots | question]; block t of the stream is encoded
    once, at its global positions S + t*B ..., against the sink alone (Eq. 4) and replaces the oldest
    block (slot t mod W).  A question attends to the sink and the blocks now in the window (Eq. 5 over the
    window); key order inside the cache does not matter to it because every key carries its own position.
    """

    def __init__(self, S, B, W, Q_max, Hq, Hkv, d, theta, scale=0.0, device="cuda"):
        import torch
        self.S, self.B, self.W, self.Q_max, self.theta, self.scale = S, B, W, Q_max, theta, scale
        self.Hq, self.Hkv, self.d = Hq, Hkv, d
        self.rows = S + W * B + Q_max
        bf, f32 = torch.bfloat16, torch.float32
        self.k_cache = torch.zeros((self.rows, Hkv, d), dtype=bf, device=device)
        self.v_cache = torch.zeros((self.rows, Hkv, d), dtype=bf, device=device)
        self.q_rows = max(S, B, Q_max)
        self.q_buf = torch.empty((self.q_rows, Hq, d), dtype=bf, device=device)
        self.s_sink = self._shape(S, 1, 0, 0)
        self.s_block = self._shape(S, B, 1, 0)
        alloc = lambda shape, dtype: torch.empty(shape, dtype=dtype, device=device)
        self.ws_sink = _workspace(alloc, pb.pevlm_workspace_bytes(self.s_sink, pb.WS_PREFILL))
        self.ws_block = _workspace(alloc, pb.pevlm_workspace_bytes(self.s_block, pb.WS_PREFILL))
        self.ws_query = _workspace(alloc, pb.pevlm_workspace_bytes(self._shape(S + W * B, 1, 0, Q_max), pb.WS_QUERY))
        self.blocks_seen = 0
        self._f32 = torch.empty((0,), dtype=f32, device=device)

    def _outputs(self, n):
        """o [n,Hq,d] and lse [Hq,n] (new_empty, which takes type and device from a tensor, costs the host half of torch.empty)."""
        return self.k_cache.new_empty((n, self.Hq, self.d)), self._f32.new_empty((self.Hq, n))

    def _shape(self, S, B, N, Q):
        return pb.make_shape(S, B, N, Q, self.Hq, self.Hkv, self.d, theta=self.theta, scale=self.scale)

    def _row(self, cache, row):
        """Address of a cache row (what cache[row:] would point to, without building the view)."""
        return cache.data_ptr() + row * self.Hkv * self.d * 2

    def set_sink(self, q, k, v):
        """Encode the sink (Eq. 3).  Returns (o [S,Hq,d], lse [Hq,S])."""
        S = self.S
        _need_rows(S, q, k, v)
        o, lse = self._outputs(S)
        pb.pevlm_rope_qkv(self.s_sink, q, k, v, self.q_buf, self.k_cache, self.v_cache, 0, S)
        pb.pevlm_parallel_prefill_attn(self.s_sink, self.q_buf, self.k_cache, self.v_cache, o, lse, self.ws_sink)
        return o, lse

    def append_block(self, q, k, v):
        """Encode the next block of the stream into the slot of the oldest one.  Returns (o [B,Hq,d], lse [Hq,B])."""
        S, B = self.S, self.B
        _need_rows(B, q, k, v)
        t = self.blocks_seen
        row0 = S + (t % self.W) * B
        o, lse = self._outputs(B)
        pb.pevlm_rope_qkv(self.s_block, q, k, v, self.q_buf, self._row(self.k_cache, row0), self._row(self.v_cache, row0), S + t * B, B)
        pb.pevlm_block_attn(self.s_block, self.q_buf, self.k_cache, self.v_cache, row0, self.rows, o, lse, self.ws_block)
        self.blocks_seen = t + 1
        return o, lse

    def ask(self, q, k, v):
        """Question of Qn <= Q_max tokens at the positions that follow the stream so far, against the sink
        and the blocks in the window (Eq. 5).  Returns (o [Qn,Hq,d], lse [Hq,Qn])."""
        Qn = q.shape[0]
        held = min(self.blocks_seen, self.W)
        nv = self.S + held * self.B
        if k.shape[0] < Qn or v.shape[0] < Qn:
            _need_rows(Qn, q, k, v)
        room = self.rows - nv  # more than Q_max while the window fills
        if Qn > room or Qn > self.q_rows:
            room = min(room, self.q_rows)
            raise ValueError(f"a question of {Qn} rows where {room} fit")
        s = self._shape(nv, 1, 0, Qn)
        o, lse = self._outputs(Qn)
        pb.pevlm_rope_qkv(s, q, k, v, self.q_buf, self._row(self.k_cache, nv), self._row(self.v_cache, nv),
                          self.S + self.blocks_seen * self.B, Qn)
        pb.pevlm_query_attn(s, self.q_buf, self.k_cache, self.v_cache, o, lse, self.ws_query)
        return o, lse

"""Where the warps of the attention kernel wait (a profiling aid, not part of the hot path).

    PEVLM_TRACE=1 python -m paper_2506_19651_b200.build --force && python -m paper_2506_19651_b200.timeline

Runs the prefill attention with a library built with the accounting of include/pevlm_trace.h, in full-causal mode on
c3_long-sized random tensors (long work items) and under the PEVLM mask (c3_long, and the 256-token blocks of the sweep:
work items of three or four key tiles), and prints, for the first pair of thread blocks, the cycles each kind of warp
spent in each kind of wait, per key tile.  The accounting itself slows the kernel by a few per cent.  Rebuild without
PEVLM_TRACE afterwards.
"""
from __future__ import annotations

import ctypes as C

import numpy as np

WAITS = {11: "Q tile", 12: "K tile", 13: "V tile", 14: "scores", 15: "probabilities", 16: "scores read", 17: "accumulator (rescale)",
         18: "probability buffer", 19: "work item", 20: "item slot", 21: "Q buffer", 22: "accumulator free", 23: "ring slot",
         25: "row sums", 26: "accumulator done", 27: "claim", 28: "hardware queue"}
ROLES = {0: "softmax 0", 4: "softmax 1", 8: "epilogue", 12: "QK issue", 14: "PV issue", 13: "producer", 15: "scheduler"}


def main():
    import torch
    from . import binding as pb, inputs
    lib = pb.lib()
    if not hasattr(lib, "pevlm_debug_waits"):
        raise SystemExit("library built without PEVLM_TRACE=1")
    for name, mode in (("c3_long", pb.MASK_FULL_CAUSAL), ("c3_long", pb.MASK_PEVLM), ("c4_sweep_F1", pb.MASK_PEVLM)):
        w = inputs.WORKLOADS[name]
        s = pb.make_shape(w.S, w.B, w.N, w.Q, w.Hq, w.Hkv, w.d, theta=w.theta, mask_mode=mode)
        nv = w.n_video
        q = torch.randn(nv, w.Hq, w.d, device="cuda", dtype=torch.bfloat16)
        k = torch.randn(nv, w.Hkv, w.d, device="cuda", dtype=torch.bfloat16)
        v = torch.randn_like(k)
        o = torch.empty_like(q)
        lse = torch.empty(w.Hq, nv, device="cuda")
        ws = torch.zeros(pb.pevlm_workspace_bytes(s, pb.WS_PREFILL), dtype=torch.uint8, device="cuda")
        for _ in range(5):
            pb.pevlm_parallel_prefill_attn(s, q, k, v, o, lse, ws)
        torch.cuda.synchronize()
        buf = (C.c_uint32 * (2 * 16 * 32))()
        assert lib.pevlm_debug_waits(buf) == 0
        t = np.array(buf, dtype=np.float64).reshape(2, 16, 32)
        tiles = t[0, 0, 1] + t[0, 4, 1]   # the two softmax warpgroups take the key tiles in turn
        print(f"-- {name}{', full causal' if mode else ''}: {tiles:.0f} key tiles, {t[0, 0, 0] / max(tiles, 1):.0f} cycles each")
        for r in range(2):
            for warp, role in ROLES.items():
                waits = ", ".join(f"{what} {t[r, warp, i] / tiles:.0f}" for i, what in WAITS.items() if t[r, warp, i] > 0)
                if waits:
                    print(f"   block {r} {role:10s} {waits}")


if __name__ == "__main__":
    main()

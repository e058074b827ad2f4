"""FP32 forward kernels at the sizes where their tiling changes: against the float64 oracle."""
import numpy as np
import pytest
import torch

import paper_2602_11562_b200 as P
from oracle import laser_oracle
from workloads import make_custom

pytestmark = pytest.mark.gpu

CASES = [
    dict(U=2, C=33, L=65, d=18, H=3, S=7, M=2, d_qh=4),              # widths that are no multiple of 4; one row past a tile
    dict(U=1, C=1, L=31, d=64, H=1, S=31, M=1),                      # 64-wide value head, four item parts, partial chunk
    dict(U=1, C=70, L=100, d=128, H=2, S=3, M=1),                    # 64-wide heads, too few items per segment to split
    dict(U=2, C=40, L=90, d=128, H=8, S=33, M=2, lengths=[90, 0]),   # eight heads, an empty user
    dict(U=3, C=400, L=64, d=32, H=2, S=16, M=2),                    # enough candidates for four per block, a partial block
    dict(U=1, C=3, L=1680, d=64, H=2, S=2, M=1),                     # segment vectors that fit only without row padding
    dict(U=1, C=5, L=40, d=256, H=4, S=20, M=1, d_qh=16),            # as many columns as threads
    dict(U=300, C=3, L=40, d=64, H=4, S=20, M=1),                    # two item parts: 2400 warps without
    dict(U=700, C=2, L=40, d=64, H=4, S=20, M=1),                    # one: 5600 warps
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_fp32_forward_edges(case):
    w = make_custom(seed=2100 + case, dtype="f32", **CASES[case])
    s = w.spec
    b = P.DeviceBatch.from_workload(w)
    ws = torch.empty(P.laser_workspace_bytes(b.cfg), dtype=torch.uint8, device="cuda")
    ws.fill_(0xFF)                                                   # (a stale status word must not survive)
    Hp, z = P.laser_forward(b.cfg, *b.args(), b.Wg, workspace=ws, want_hprime=True)
    assert P.laser_check_status(ws) == 0
    Hr, zr = laser_oracle.forward(w.items, w.lengths, w.cands, w.cand_offsets, w.Wq, w.Wk, w.Wv, w.Wg, s.S, s.H, w.gamma, w.tau)
    for got, ref in ((Hp, Hr), (z, zr)):
        g = got.cpu().numpy().astype(np.float64)
        assert np.isfinite(g).all() and np.max(np.abs(g - ref) / np.maximum(1.0, np.abs(ref))) <= 1e-4

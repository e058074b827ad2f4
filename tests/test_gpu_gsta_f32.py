"""The fp32 stacked-attention kernel for compile-time widths: every (width, heads), the candidate counts at which the number of
candidates per block changes, partial blocks, users without items or candidates; after the whole forward and on its own."""
import numpy as np
import pytest
import torch

import paper_2602_11562_b200 as P
from oracle import laser_oracle
from workloads import make_custom

pytestmark = pytest.mark.gpu

WIDTHS = [(32, 1), (32, 2), (64, 1), (64, 2), (64, 4), (96, 3), (96, 6), (128, 1), (128, 2), (128, 4), (128, 8)]


def _case(d, H, U, C, L, S, M, dtype, seed, lengths=None):
    w = make_custom(U=U, C=C, L=L, d=d, H=H, S=S, M=M, d_qh=16, dtype=dtype, seed=seed, emb_std="inv_sqrt_d", lengths=lengths)
    s = w.spec
    b = P.DeviceBatch.from_workload(w, path=P.PATH_SIMT)
    ws = torch.empty(P.laser_workspace_bytes(b.cfg), dtype=torch.uint8, device="cuda")
    ws.fill_(0xFF)
    Hp, z = P.laser_forward(b.cfg, *b.args(), b.Wg, workspace=ws, want_hprime=True)
    assert P.laser_check_status(ws) == 0
    z2 = P.laser_gsta_forward(b.cfg, Hp, b.lengths, b.cand_offsets, b.cands, b.Wg, workspace=ws)
    assert P.laser_check_status(ws) == 0 and torch.equal(z, z2)
    # the reference runs on the kernel's own H' (in bf16 its rounding is not this kernel's)
    H64 = Hp.float().cpu().numpy().astype(np.float64)
    ref = laser_oracle.gsta_forward(H64, w.lengths, w.cand_offsets, w.cands, w.Wg, s.S, s.H, w.tau)
    got = z.float().cpu().numpy().astype(np.float64)
    # fp32: sums of up to 128 + 128 products per step, a few layers: 2^-24 sqrt(256) per step and margin; bf16 rounds z once (2^-9)
    tol = 2e-5 if dtype == "f32" else 2.0 ** -8
    assert np.isfinite(got).all()
    assert np.max(np.abs(got - ref) / np.maximum(1.0, np.abs(ref))) <= tol


@pytest.mark.parametrize("d,H", WIDTHS)
def test_every_width(d, H):
    _case(d, H, U=3, C=7, L=70, S=9, M=2, dtype="f32", seed=31, lengths=[70, 0, 33])
    _case(d, H, U=2, C=5, L=40, S=40, M=3, dtype="bf16", seed=32, lengths=[40, 1])


@pytest.mark.parametrize("N", [296, 297, 888, 889, 891])
@pytest.mark.parametrize("d,H", [(64, 4), (96, 3), (128, 8)])
def test_candidates_per_block(d, H, N):
    _case(d, H, U=1, C=N, L=60, S=4, M=1, dtype="f32", seed=33)


def test_many_segments():
    _case(128, 8, U=1, C=300, L=300, S=3, M=1, dtype="f32", seed=34)       # 100 segments: two candidates take 139 KB
    _case(128, 2, U=1, C=3, L=1200, S=3, M=1, dtype="f32", seed=35)        # 400 segments: more than one block's shared memory
    _case(64, 2, U=2, C=900, L=500, S=5, M=1, dtype="bf16", seed=36, lengths=[500, 499])

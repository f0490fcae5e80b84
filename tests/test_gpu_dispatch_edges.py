"""Parity at the sizes where a dispatch rule changes its mind or a tile is ragged: one row past a tile, the last size of a
split, head counts that are not powers of two.  Tolerances are those of the files that cover the same entry points."""
import numpy as np
import pytest
import torch

from oracle import dsla_oracle as orc

pytestmark = pytest.mark.gpu
BF = torch.bfloat16


# split 8 (few tiles), 4 (19..37 tiles), 2 (38..74), none; H = 40: twenty 16-byte pieces per row; H = 8: four
@pytest.mark.parametrize("T,H,D_model", [(127, 40, 2048), (18 * 128 + 1, 8, 2048), (37 * 128, 16, 1024), (38 * 128 - 1, 24, 512),
                                         (75 * 128 - 5, 8, 512), (200, 96, 1024)])
def test_gate_project_cluster_splits(T, H, D_model):
    import paper_2506_09316_b200 as dsla
    rng = np.random.default_rng(5100 + T)
    x = torch.from_numpy(rng.normal(size=(T, D_model)).astype(np.float32)).to(BF)
    w = torch.from_numpy((rng.normal(size=(2 * H, D_model)) * (2.0 / np.sqrt(D_model))).astype(np.float32)).to(BF)
    b = torch.from_numpy(rng.normal(size=2 * H).astype(np.float32) * 2.0)
    band = 64
    gh, gr = (torch.full((T + band, H), 7.0, device="cuda") for _ in range(2))
    for _ in range(2):          # back to back: the second launch overlaps the first one's tail
        dsla.dsla_gate_project(x.cuda(), w.cuda(), b.cuda(), g_hist=gh[:T], g_rec=gr[:T])
    torch.cuda.synchronize()
    assert dsla.dsla_gate_project_last_error() == dsla.DSLA_OK
    rows = np.unique(np.concatenate([np.arange(min(T, 160)), np.arange(max(0, T - 160), T)]))
    ref = orc.gate_project(x[rows].double().numpy(), w.double().numpy().T, b.double().numpy())
    got = np.concatenate([gh[:T].double().cpu().numpy()[rows], gr[:T].double().cpu().numpy()[rows]], axis=1)
    assert np.max(np.abs(got - ref)) <= 2e-5
    assert bool((gh[:T] <= 1.0).all()) and bool((gr[:T] <= 1.0).all())      # every row written
    assert bool((gh[T:] == 7.0).all()) and bool((gr[T:] == 7.0).all())      # and none past the end

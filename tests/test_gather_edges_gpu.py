"""Row gathers where their index arithmetic can go wrong: rows of 1 to 3 vectors and of odd counts, batch items that
begin and end inside a block of 1024 vectors or span several, more batch items in a block than one."""
import numpy as np
import pytest
import torch

from oracle import hilberta_oracle as orc
from paper_2509_26538_b200 import binding as hb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,text,batch,vecs", [
    (8, 8, 0, 1, 1), (8, 8, 0, 33, 1), (8, 8, 3, 700, 1),       # 67 vectors an item: up to 16 items in a block
    (2, 2, 0, 1000, 1), (1, 1, 0, 1500, 3),                     # items of 4 and 3 vectors
    (16, 16, 0, 5, 4), (32, 32, 0, 3, 1),                       # an item is a block exactly
    (17, 23, 5, 4, 3), (31, 9, 1, 7, 17), (40, 24, 77, 2, 129), (64, 64, 33, 1, 383),
])
def test_gather_edges(H, W, text, batch, vecs):
    plan = hb.Plan(H, W, 1, 0, 0, text)
    S = text + H * W
    to_orig = orc.plan_arrays(H, W, 1, 0, 0, text)["phys2orig"]
    x = torch.arange(batch * S * vecs * 4, dtype=torch.float32, device="cuda").view(batch, S, vecs * 4)
    guard = torch.full((x.numel() + 64,), -1.0, device="cuda")
    y = guard[32:-32].view_as(x)
    plan.permute(x, y)
    assert torch.equal(y, x[:, torch.from_numpy(np.asarray(to_orig)).long().cuda()])
    assert (guard[:32] == -1).all() and (guard[-32:] == -1).all()
    z = torch.empty_like(x)
    plan.unpermute(y, z)
    assert torch.equal(z, x)
    plan.destroy()

"""The tiled form of the allocation-free iteration against the regular tree mode, bit for
bit: one particle, tiles of padding only, ragged tiles and dimensions, the widest
particle, and both sides of the line to the tree step."""
import numpy as np
import pytest

from tests.gpu_common import BOUNDS, C12, W, load_cupso, same_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fid,N,D,pad", [(0, 1, 1, 0), (2, 130, 3, 2048), (3, 777, 33, 0), (1, 300, 1024, 128),
                                         (4, 262144, 2, 0), (1, 262145, 2, 0), (2, 40000, 20, 0)])
def test_noalloc_equals_tree_mode(fid, N, D, pad):
    P = load_cupso()
    import torch
    ld, seed = (N + 127) // 128 * 128 + pad, 7
    lo, hi, vmax = b = (0.0, 3.0, 0.5) if fid == 4 else BOUNDS[fid]      # a zero bound: the general clamps
    with P.Swarm(D, N, b, W, C12, C12, fid, seed, mode="tree") as s:
        st, g = s.state(), s.gbest()
        s.step(3)
        ref, gref = s.state(), s.gbest()

    def plane(a):
        out = torch.full((D, ld), 0.5, device="cuda")
        out[:, :N] = torch.from_numpy(np.ascontiguousarray(a.T)).cuda()
        return out

    x, v, pb = plane(st["pos"]), plane(st["v"]), plane(st["pbest_pos"])
    pf = torch.zeros(ld, device="cuda")                                  # padding with the best fitness of all
    pf[:N] = torch.from_numpy(st["pbest_fit"]).cuda()
    gp = torch.from_numpy(g[3].copy()).cuda()
    gf, gi = torch.empty(1, device="cuda"), torch.empty(1, dtype=torch.int64, device="cuda")
    pad_x, pad_pb = x[:, N:].clone(), pb[:, N:].clone()
    for t in (1, 2, 3):
        P.cupso_tree_step_noalloc(D, N, b, W, C12, C12, fid, seed, 0, t, x.data_ptr(), v.data_ptr(), pb.data_ptr(),
                                  pf.data_ptr(), ld, gp.data_ptr(), gf.data_ptr(), gi.data_ptr(), 0,
                                  torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    for name, a in (("pos", x), ("v", v), ("pbest_pos", pb)):
        assert same_bits(a[:, :N].T.cpu().numpy(), ref[name]), name
    assert same_bits(pf[:N].cpu().numpy(), ref["pbest_fit"])
    assert same_bits(gp.cpu().numpy(), gref[3]) and int(gi.item()) == gref[2] and gf.item() == gref[1]
    if ld > N:                                                           # moved, but never improved
        assert not torch.equal(x[:, N:], pad_x) and torch.equal(pb[:, N:], pad_pb)

"""Routing from a given mask: the entry that copies the mask and the one that finds it in place give what the oracle gives, whatever the
buffers held before."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_2310_04361_b200 import api
    return api


# both sides of: one CTA (64), one launch (1024), counts added up by every CTA (16384 of them); ragged last blocks, words and experts
@pytest.mark.parametrize("T,E,p", [(1, 24, 0.5), (64, 24, 0.1), (65, 24, 0.1), (256, 5, 0.0), (1024, 32, 0.3), (1025, 32, 1.0), (1300, 33, 0.2),
                                   (3001, 344, 0.05), (12289, 344, 0.02), (50433, 24, 0.1), (50432, 128, 0.02)])
def test_mask_routing(api, T, E, p):
    rng = np.random.default_rng(T + E)
    G = (rng.random((T, E)) < p).astype(np.uint8)
    words = torch.from_numpy(oracle.pack_mask(G).view(np.int32)).cuda()
    want = oracle.metadata(G)
    dirty = torch.full((T * E * 2,), -3, dtype=torch.int32, device="cuda")      # what the allocator hands out next
    del dirty
    in_place = api.Routing(T, E, words.device)
    in_place.mask.copy_(words)
    ws = torch.full((max(int(api._lib.d2d_select_workspace_bytes(T, E)), 256),), 0x55, dtype=torch.uint8, device="cuda")
    api._check(api._lib.d2d_routing_from_mask(T, E, api.ctypes.byref(in_place.struct), ws.data_ptr(), ws.numel(), api._stream()), "from_mask")
    for r in (api.routing_from_mask(words, E), in_place):
        assert r.status == 0 and r.n_sel == int(G.sum())
        assert np.array_equal(r.mask_u32(), oracle.pack_mask(G))
        assert np.array_equal(r.k[:T].cpu().numpy(), G.sum(1))
        assert np.array_equal(r.counts.cpu().numpy(), want["counts"])
        assert np.array_equal(r.offsets.cpu().numpy(), want["offsets"])
        assert np.array_equal(r.perm[: r.n_sel].cpu().numpy(), want["perm"])
        assert not r.perm[r.n_sel:].any()


def test_capacity_and_strided_masks(api):
    T, E = 2000, 24
    words = torch.randint(0, 1 << 24, (T, 2), dtype=torch.int32, device="cuda")[:, :1]      # not contiguous: copied first
    a, b = api.routing_from_mask(words, E), api.routing_from_mask(words.contiguous(), E)
    assert torch.equal(a.mask, b.mask) and torch.equal(a.perm, b.perm) and a.n_sel == b.n_sel
    r = api.Routing(T, E, words.device, perm_capacity=100)
    r._slab.fill_(-7)
    src, ws = words.contiguous(), torch.empty((1 << 16,), dtype=torch.uint8, device="cuda")
    api._check(api._lib.d2d_routing_of_mask(src.data_ptr(), T, E, api.ctypes.byref(r.struct), ws.data_ptr(), ws.numel(), api._stream()), "of_mask")
    assert r.status == 7 and r.n_sel == a.n_sel and torch.equal(r.perm[:100], a.perm[:100])
    at = r._shapes["perm"][2] + 100
    assert r._slab[at:].numel() == 28 and bool((r._slab[at:] == -7).all())      # the padding behind perm

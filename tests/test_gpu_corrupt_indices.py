"""Sums of payloads whose indices are corrupt (they do not ascend, or lie beyond the bucket): reported, whatever the workspace
held before, and summed as far as they are in order."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2506_16235_b200 as nsml

SMALL, LARGE = 300_001, 3_000_001  # tiles of 2048 and 8192


def tile_of(n):
    return 2048 if n <= 1 << 21 else 8192


def sum_of(n, idx, fill):
    """(status, dense, offset table) of a sum of one payload with these indices, all values 1."""
    idx = np.asarray(idx, dtype=np.uint32)
    raw = nsml.pack_payload(n, 32, np.arange(idx.size, dtype=np.uint32), f32=np.ones(idx.size, np.float32))
    raw[64:64 + 4 * idx.size] = idx.view(np.uint8)
    payload, dense = torch.from_numpy(raw).cuda(), torch.zeros(n, device="cuda")
    ws = torch.full((nsml.nsml_accumulate_workspace_bytes(n, 1),), fill, dtype=torch.uint8, device="cuda")
    nsml.nsml_decompress_accumulate([payload], dense, workspace=ws)
    tiles = (n + tile_of(n) - 1) // tile_of(n)
    status = nsml.nsml_last_status(ws)
    return status, dense, ws[256:256 + 4 * (tiles + 1)].view(torch.int32).cpu().numpy().view(np.uint32)


def corrupt(n, kind, k, rng):
    idx = np.sort(rng.choice(n, k, replace=False))
    if kind == "swapped":  # two entries of different tiles
        idx[[k // 3, 2 * k // 3]] = idx[[2 * k // 3, k // 3]]
    elif kind == "shuffled":
        rng.shuffle(idx)
    elif kind == "descending":
        idx = idx[::-1]
    elif kind == "first last":
        idx[[0, -1]] = idx[[-1, 0]]
    elif kind == "middle beyond":  # behind the last tile, then back
        idx[k // 2] = 0xFFFFFFF0
    elif kind == "last beyond":
        idx[-1] = 0xFFFFFFF0
    elif kind == "end beyond":  # ascending, the last few behind the last tile
        idx[-5:] = ((n + tile_of(n) - 1) // tile_of(n)) * tile_of(n) + np.arange(5)
    elif kind == "inside the last tile":  # behind the bucket, but not behind its last tile
        idx[-1] = n
    return idx


# 120000 entries are read as a whole, 2000000 are more than the partition's blocks read: boundaries are searched
@pytest.mark.parametrize("n,k", [(SMALL, 4), (SMALL, 5), (SMALL, 5000), (LARGE, 120_000), (LARGE, 2_000_000)])
@pytest.mark.parametrize("kind", ["swapped", "shuffled", "descending", "first last", "middle beyond", "last beyond", "end beyond", "inside the last tile"])
def test_reported_whatever_the_workspace_held(n, k, kind):
    if kind == "end beyond" and k < 10:
        k += 6
    idx = corrupt(n, kind, k, np.random.default_rng(k))
    for fill in (0x00, 0xFF, 0x55):
        status, _, table = sum_of(n, idx, fill)
        assert int(table.max()) <= k, "a boundary was not written"
        assert table[0] == 0 and status == nsml.NSML_ERR_PAYLOAD


@pytest.mark.parametrize("n,k", [(SMALL, 5000), (LARGE, 120_000)])
def test_order_inside_a_tile_does_not_matter(n, k):
    rng = np.random.default_rng(3)
    idx = np.sort(rng.choice(n, k, replace=False))
    order = np.lexsort((rng.random(k), idx // tile_of(n)))
    for fill in (0x00, 0xFF):
        status, dense, _ = sum_of(n, idx[order], fill)
        want = torch.zeros(n, device="cuda")
        want[torch.from_numpy(idx).cuda()] = 1.0
        assert status == 0 and torch.equal(dense, want)

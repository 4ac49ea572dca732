"""The culling kernel's parts of several 256-slot chunks (large inputs): chunks that begin exactly
where a record ends, the slot cache and its absence, lists that overflow, and more chunks than
the table of first records holds.  A slot is one tile row of a visible record's rectangle."""
import numpy as np
import pytest
import torch

import synthetic
from test_gpu_parity import _check_ranges_and_order, _gpu_lists, f32_camera, lists_match_kernel_rule, make

pytestmark = pytest.mark.gpu


def _scene(N, W, H, f, sx, sy, seed):
    """N Gaussians before an identity camera, their means spread over the image, with standard
    deviations of about sx x sy pixels (before any rotation: sy None turns them at random)."""
    rng = np.random.default_rng(seed)
    z = rng.uniform(1.0, 3.0, N)
    u, v = rng.uniform(0, W - 1, N), rng.uniform(0, H - 1, N)
    mean = np.stack([(u - (W / 2 - 0.5)) / f * z, (v - (H / 2 - 0.5)) / f * z, z], 1)
    s = np.stack([rng.uniform(*sx, N), rng.uniform(*(sy or sx), N), rng.uniform(*sx, N)], 1) * (z / f)[:, None]
    q = rng.normal(size=(N, 4)) if sy is None else np.tile([1.0, 0.0, 0.0, 0.0], (N, 1))
    a = lambda x: np.ascontiguousarray(x, dtype=np.float32)
    g = dict(mean=a(mean), log_scale=a(np.log(s)), quat=a(q / np.linalg.norm(q, axis=1, keepdims=True)),
             opacity_logit=a(rng.normal(0.5, 1.0, N)), rgb=a(rng.uniform(0, 1, (N, 3))), sem=a(np.zeros((N, 4))))
    return g, f32_camera(synthetic.make_camera(W, H, f, f, W / 2 - 0.5, H / 2 - 0.5))


def _slots(r):
    rect = r.rect.view(-1, 2).cpu().numpy().view(np.uint32).astype(np.int64)
    rows = (rect[:, 1] >> 16) - (rect[:, 0] >> 16)
    cols = (rect[:, 1] & 0xFFFF) - (rect[:, 0] & 0xFFFF)
    return np.where((rows > 0) & (cols > 0), rows, 0)


def _several_chunks(slots):
    """Whether a part holds several chunks: there are at most two parts per block and six blocks
    per SM."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return slots > 2 * 6 * sms * 256


@pytest.mark.parametrize("tile, half", [((8, 8), False), ((8, 8), True), ((16, 16), False)])
def test_chunks_of_256_one_row_records(tile, half):
    """An image of one tile row: every chunk's 256 slots belong to 256 records, and each chunk
    begins in another record than the chunk before it ends in."""
    g, cam = _scene(1_200_000, 4096, 8, 1000.0, (0.3, 1.2), None, 1)
    r, p = make(g, [cam], capacity=1 << 23, tile_w=tile[0], tile_h=tile[1], half_masks=half)
    r.project(p)
    rows = _slots(r)
    assert rows.max() == 1 and _several_chunks(int(rows.sum()))
    r.build_lists()
    assert lists_match_kernel_rule(r) > 1_000_000


@pytest.mark.parametrize("half", [False, True])
def test_parts_of_several_chunks_at_every_capacity(half):
    """Capacity for everything (the lists of the kernels' rule); below the instances, with and
    without room for the slot cache: the first `capacity` instances of the emission order (depth,
    record, tile), sorted by tile."""
    g, cam = _scene(150_000, 1024, 768, 500.0, (1.0, 9.0), None, 2)
    kw = dict(tile_w=8, tile_h=8, half_masks=half)
    r, p = make(g, [cam], capacity=1 << 23, **kw)
    r.project(p)
    slots = int(_slots(r).sum())
    assert _several_chunks(slots)
    r.build_lists()
    K = lists_match_kernel_rule(r)
    assert slots + 1000 < K
    _, tiles, recs, _ = _gpu_lists(r)
    words = r.record[:K].cpu().numpy().view(np.uint32)
    depth = r.geo.view(-1, 8)[:, 2].contiguous().view(torch.int32).cpu().numpy()[recs]
    emitted = np.lexsort((tiles, recs, depth))
    for cap in (K - 1, slots + 999, slots, slots - 1, slots // 2, 5000):
        r2, p2 = make(g, [cam], capacity=cap, **kw)
        r2.project(p2)
        r2.build_lists()
        torch.cuda.synchronize()
        assert int(r2.status.item()) & 1 and r2.instance_count() == K
        first = emitted[:cap]
        want = first[np.argsort(tiles[first], kind="stable")]
        assert np.array_equal(r2.tile[:cap].cpu().numpy().view(np.uint32), tiles[want])
        assert np.array_equal(r2.record[:cap].cpu().numpy().view(np.uint32), words[want])
        _check_ranges_and_order(r2, tiles[want], r2.ranges.view(-1, 2).cpu().numpy().astype(np.int64))


def test_more_chunks_than_the_table_of_first_records():
    """Over 65536 chunks of 256 slots (records of some 260 tile rows): the union of the lists of
    both halves of the records, each within the table."""
    N = 90_000
    g, cam = _scene(N, 64, 2100, 500.0, (0.3, 0.8), (900.0, 1500.0), 3)

    def lists(a, b):
        r, p = make({k: v[a:b] for k, v in g.items()}, [cam], capacity=48 << 20, tile_w=8, tile_h=8)
        r.project(p)
        r.build_lists()
        torch.cuda.synchronize()
        assert int(r.status.item()) == 0
        K, slots = r.instance_count(), int(_slots(r).sum())
        tile, rec = r.tile[:K].long(), r.record[:K].long()
        return slots, tile, rec + a, tile << 32 | r.geo.view(-1, 8)[:, 2].contiguous().view(torch.int32)[rec].long()

    slots, tile, rec, key = lists(0, N)
    assert slots > 65536 * 256
    parts = [lists(0, N // 2), lists(N // 2, N)]
    assert all(p[0] < 65536 * 256 for p in parts)
    want, order = torch.cat([p[3] for p in parts]).sort(stable=True)
    assert torch.equal(key, want)
    assert torch.equal(rec, torch.cat([p[2] for p in parts])[order])

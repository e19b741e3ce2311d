"""GPU: the queued 3D kernels (dense and sparse grids, deterministic and stochastic) and the
kernels that take their calls without a queue, at the sizes and
positions where their queues can go wrong: partly filled warps and chunks, misaligned
arrays, calls on either side of the 128-query chunk limit, windows on the grid's edges,
across leaves, lower and upper nodes, and next to voxels that are not finite."""
import numpy as np
import pytest
import torch

import paper_2305_05810_gb300 as stf
import synth
from oracle import filters, textures
from parity import abs_weighted_sum, check_deterministic, dev, quantise, to_dev
from test_gpu_sparse_binning import sparse_pair

pytestmark = pytest.mark.gpu
FILTERS = ["linear", "bspline3", "catmull_rom"]
CHUNKED = 1 << 20          # calls of at least this many queries take 128-query chunks
SPECIAL = [[np.nan, 1, 1], [np.inf, 2, 2], [1, -np.inf, 2], [1e9, 1, 1], [-3e38, 0, 0],
           [2.0 ** 24, 3, 3], [-2.0 ** 24, 3, 3]]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    stf.load()


def _points(n, lo, hi, seed):
    """Points inside and around [lo, hi), integer ones and special ones among them."""
    span = np.float32(hi - lo)
    p = synth.uniform(3 * n, seed).reshape(-1, 3) * (span * np.float32(1.5)) + np.float32(lo) - span / np.float32(4)
    p[::7] = np.floor(p[::7])
    k = min(n, len(SPECIAL))
    p[n // 2:n // 2 + k] = np.array(SPECIAL, dtype=np.float32)[:len(p[n // 2:n // 2 + k])]
    return p.astype(np.float32)


def _dense(fmt, dims=(23, 18, 21), background=0.25):
    x, y, z = dims
    v = synth.uniform(x * y * z, 4).reshape(z, y, x)
    T = stf.Texture(stf.KIND_DENSE3D, v, dims=dims, fmt=fmt, background=background)
    return T, textures.Dense3D(quantise(v, fmt), background)


def _sparse(fmt, background=0.25):
    """Leaves with gaps around the corner of four lower nodes and of two upper nodes."""
    g = np.stack(np.meshgrid(*[np.arange(-4, 4)] * 3, indexing="ij"), -1).reshape(-1, 3)
    keep = synth.uniform(len(g), 9) < 0.6
    origins = (g[keep] * 8 + np.array([128, 0, 4096])).astype(np.int32)
    values = synth.uniform(512 * len(origins), 10).reshape(-1, 512) + np.float32(0.1)
    return sparse_pair(origins, values, fmt, background)


def _check(T, ref, pts, filt):
    det = T.lookup_deterministic(to_dev(pts), filter=filt).cpu().numpy()
    dv, _, _ = filters.lookup_3d(ref, pts, filt, stochastic_form=False)
    scale = abs_weighted_sum(ref.fetch, [pts[:, 0], pts[:, 1], pts[:, 2]], filt)
    check_deterministic(det, dv, np.maximum(np.nan_to_num(scale), abs(ref.background)))


@pytest.mark.parametrize("fmt", [stf.FMT_F16, stf.FMT_F32])
@pytest.mark.parametrize("filt", FILTERS)
def test_dense_edges_match_oracle(filt, fmt):
    T, ref = _dense(fmt)
    for n in (1, 31, 33, 4099):
        _check(T, ref, _points(n, 0, 23, n), filt)


@pytest.mark.parametrize("dims", [(1, 1, 1), (2, 3, 1), (5, 4, 4), (64, 4, 5)])
def test_dense_small_grids_match_oracle(dims):
    T, ref = _dense(stf.FMT_F16, dims)
    _check(T, ref, _points(2000, 0, max(dims), 3), "bspline3")


@pytest.mark.parametrize("fmt", [stf.FMT_F32, stf.FMT_E4M3_SCALED])
@pytest.mark.parametrize("filt", FILTERS)
def test_sparse_nodes_match_oracle(filt, fmt):
    T, ref = _sparse(fmt)
    for n in (1, 31, 33, 4099):
        p = _points(n, -32, 32, n)
        p[np.abs(p[:, 0]) < 1000] += np.array([128, 0, 4096], dtype=np.float32)
        _check(T, ref, p, filt)
    stf.stf_synchronize(T.handle)


@pytest.mark.parametrize("kind", ["dense", "sparse"])
@pytest.mark.parametrize("shift", [0, 1])
def test_chunk_sizes_and_alignment_give_the_same_bits(kind, shift):
    """One large call (128-query chunks; aligned and misaligned arrays, a ragged end)
    equals the same queries in small calls (32-query chunks)."""
    T, _ = _dense(stf.FMT_F16) if kind == "dense" else _sparse(stf.FMT_E4M3_SCALED)
    n = CHUNKED + 77
    p = _points(n, 0, 23, 5) if kind == "dense" else _points(n, -32, 32, 5) + np.array([128, 0, 4096], np.float32)
    buf = torch.empty((n + 1, 3), dtype=torch.float32, device=dev())
    c = buf[shift:shift + n]
    c.copy_(to_dev(p))
    out = torch.full((n + 1, 1), 7.0, device=dev())
    T.lookup_deterministic(c, out=out[shift:shift + n], filter="bspline3")
    parts = [T.lookup_deterministic(c[i:i + 300001].clone(), filter="bspline3") for i in range(0, n, 300001)]
    torch.testing.assert_close(out[shift:shift + n], torch.cat(parts), rtol=0, atol=0)
    assert float(out[0 if shift else n]) == 7.0


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("fmt", [stf.FMT_F16, stf.FMT_F32])
def test_dense_neighbours_of_non_finite_voxels_are_not_read(fmt, bad):
    """Rows are loaded in wider aligned words than a window: voxels outside the window,
    finite or not, must not reach the result."""
    v = synth.uniform(16 ** 3, 4).reshape(16, 16, 16)
    w = v.copy()
    w[8, 8, 8] = bad
    p = synth.uniform(3 * 20000, 6).reshape(-1, 3) * np.float32(16)
    a, b = (stf.Texture(stf.KIND_DENSE3D, t, dims=(16, 16, 16), fmt=fmt).lookup_deterministic(
        to_dev(p), filter="bspline3").cpu().numpy()[:, 0] for t in (v, w))
    base = np.floor(p)
    touched = np.all((base >= 6) & (base <= 9), axis=1)     # 8 in [base - 1, base + 2] on every axis
    assert np.array_equal(a[~touched], b[~touched])
    assert not np.isfinite(b[touched]).any() and touched.any()


def test_sparse_neighbours_of_non_finite_voxels_are_not_read():
    origins = np.stack(np.meshgrid(*[np.arange(2) * 8] * 3, indexing="ij"), -1).reshape(-1, 3).astype(np.int32)
    v = synth.uniform(512 * 8, 4).reshape(8, 512)
    w = v.copy()
    w[0, 5 * 64 + 5 * 8 + 5] = np.nan                        # voxel (5, 5, 5) of the leaf at the origin
    p = synth.uniform(3 * 20000, 6).reshape(-1, 3) * np.float32(14)
    a, b = (stf.Texture(stf.KIND_SPARSE3D, t, fmt=stf.FMT_F32, leaf_origins=origins).lookup_deterministic(
        to_dev(p), filter="bspline3").cpu().numpy()[:, 0] for t in (v, w))
    base = np.floor(p)
    touched = np.all((base >= 3) & (base <= 6), axis=1)
    assert np.array_equal(a[~touched], b[~touched])
    assert np.isnan(b[touched]).all() and touched.any()


@pytest.mark.parametrize("filt", ["linear", "bspline3", "fis_linear", "fis_bspline3"])
@pytest.mark.parametrize("kind", ["dense", "sparse"])
def test_stochastic_queue_equals_the_general_loop(kind, filt):
    """Queued stochastic calls (chunks of 32 and of 128; aligned and misaligned arrays; ragged
    ends; few, most and no queries live; counters that cross 2^32) against the call with tap
    output, which takes the general loop."""
    T, _ = _dense(stf.FMT_F16) if kind == "dense" else _sparse(stf.FMT_E4M3_SCALED)
    for n, spread in ((1, 1.0), (33, 1.0), (4099, 1.0), (CHUNKED + 77, 1.0), (CHUNKED + 77, 0.01), (CHUNKED, 100.0)):
        p = _points(n, 0, 23, 5) if kind == "dense" else _points(n, -32, 32, 5)
        p = p * np.float32(spread)
        p = (p + (np.float32(8) if kind == "dense" else np.array([128, 0, 4096], np.float32))).astype(np.float32)
        for shift in (0, 1):
            buf = torch.empty((n + 1, 3), dtype=torch.float32, device=dev())
            c = buf[shift:shift + n]
            c.copy_(to_dev(p))
            out = torch.full((n + 1, 1), 7.0, device=dev())
            args = dict(filter=filt, seed=11, query_offset=(1 << 32) - 1000)
            T.lookup(c, out=out[shift:shift + n], **args)
            want = T.lookup(c, taps=torch.empty((n, 4), dtype=torch.int32, device=dev()), **args)
            torch.testing.assert_close(out[shift:shift + n], want, rtol=0, atol=0)
            assert float(out[0 if shift else n]) == 7.0


@pytest.mark.parametrize("filt", ["linear", "bspline3"])
@pytest.mark.parametrize("kind", ["dense", "sparse"])
def test_arrays_in_host_memory_give_the_same_bits(kind, filt):
    """Coordinates, results or both in page-locked memory, which take the kernels without a
    queue."""
    T, _ = _dense(stf.FMT_F16) if kind == "dense" else _sparse(stf.FMT_E4M3_SCALED)
    for n in (33, 4099, CHUNKED + 77):
        p = _points(n, 0, 23, 5) if kind == "dense" else _points(n, -32, 32, 5) + np.array([128, 0, 4096], np.float32)
        c = to_dev(p.astype(np.float32))
        host = torch.empty((n, 3), pin_memory=True)
        host.copy_(c)
        for look in (lambda x, out=None: T.lookup_deterministic(x, filter=filt, out=out),
                     lambda x, out=None: T.lookup(x, filter=filt, seed=3, out=out)):
            want = look(c)
            out = torch.full((n, 1), 7.0, device=dev())
            look(host, out)
            torch.testing.assert_close(out, want, rtol=0, atol=0)
            for x in (c, host):
                out = torch.full((n, 1), 7.0, pin_memory=True)
                look(x, out)
                stf.stf_synchronize(T.handle)
                torch.testing.assert_close(out, want.cpu(), rtol=0, atol=0)


@pytest.mark.parametrize("filt", ["linear", "bspline3", "fis_bspline3"])
@pytest.mark.parametrize("kind", ["dense", "sparse"])
def test_calls_taken_directly_and_by_queue(kind, filt):
    """Calls of whose queries three quarters are live are taken without the queue, judged by a
    few of them: the same bits for any share and place of the live ones."""
    T, _ = _dense(stf.FMT_F16) if kind == "dense" else _sparse(stf.FMT_E4M3_SCALED)
    for n in (CHUNKED, CHUNKED + 77):
        i, u = np.arange(n), synth.uniform(n, 6)
        p = synth.uniform(3 * n, 5).reshape(-1, 3) * np.float32(14)
        p += np.float32(4) if kind == "dense" else np.array([124, -4, 4092], np.float32)
        for live in (i >= 0, u < 0.8, u < 0.75, u < 0.7, i < n // 2, i >= n // 2, i % 128 < 100):
            x = p.copy()
            x[~live] = -1e5
            x[::1001] = np.nan
            c = to_dev(x)
            args = dict(filter=filt, seed=11, query_offset=(1 << 32) - 1000)
            want = T.lookup(c, taps=torch.empty((n, 4), dtype=torch.int32, device=dev()), **args)
            torch.testing.assert_close(T.lookup(c, **args), want, rtol=0, atol=0)

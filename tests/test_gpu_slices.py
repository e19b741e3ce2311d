"""GPU: calls of more than 2^30 queries, which the kernels with 32-bit query indices take in
slices: the queries on both sides of a slice's end have the bits that they have in a small
call."""
import pytest
import torch

import paper_2305_05810_gb300 as stf
import synth
from parity import dev
from test_gpu_queue import _dense, _sparse

pytestmark = pytest.mark.gpu
SLICE = 1 << 30
N, K = SLICE + 3001, 6001           # the last K queries are looked at, SLICE among them


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.mem_get_info()[0] < 48 << 30:
        pytest.skip("needs 48 GB of device memory")
    stf.load()
    yield
    torch.cuda.empty_cache()


def _batch(tail, fill):
    a = torch.full((N,) + tail.shape[1:], fill, device=dev())
    a[N - K:] = tail
    return a


def _same(out, want):
    torch.testing.assert_close(out[N - K:], want, rtol=0, atol=0)


@pytest.mark.parametrize("kind", ["dense", "sparse"])
def test_deterministic_grid(kind):
    T, _ = _dense(stf.FMT_F16) if kind == "dense" else _sparse(stf.FMT_E4M3_SCALED)
    tail = torch.from_numpy(synth.uniform(3 * K, 5).reshape(-1, 3)).to(dev()) * 20
    if kind == "sparse":
        tail = tail + torch.tensor([120.0, -8.0, 4088.0], device=dev())
    _same(T.lookup_deterministic(_batch(tail, -1e5), filter="bspline3"), T.lookup_deterministic(tail, filter="bspline3"))


@pytest.mark.parametrize("levels", [1, 7])
def test_deterministic_cubic_image(levels):
    T = stf.Texture(stf.KIND_TEX2D, synth.texture2d(64, 64, 1, seed=3), dims=(64, 64, 1), mip_levels=levels,
                    generate_mips=levels > 1)
    tail = torch.from_numpy(synth.uniform(2 * K, 8).reshape(-1, 2)).to(dev())
    lod = None if levels == 1 else torch.from_numpy(synth.uniform(K, 9)).to(dev()) * 6
    _same(T.lookup_deterministic(_batch(tail, 0.5), None if lod is None else _batch(lod, 0.0), filter="bspline3"),
          T.lookup_deterministic(tail, lod, filter="bspline3"))


def test_ewa():
    T = stf.Texture(stf.KIND_TEX2D, synth.texture2d(64, 64, 1, seed=3), dims=(64, 64, 1), mip_levels=7, generate_mips=True)
    tail = torch.from_numpy(synth.uniform(2 * K, 8).reshape(-1, 2)).to(dev())
    grad = (torch.from_numpy(synth.uniform(4 * K, 9).reshape(-1, 4)).to(dev()) - 0.5) * 0.1
    uv, g = _batch(tail, 0.5), _batch(grad, 0.0)
    _same(T.lookup_ewa_deterministic(uv, g), T.lookup_ewa_deterministic(tail, grad))
    taps = torch.zeros((N, 4), dtype=torch.int32, device=dev())
    small = torch.zeros((K, 4), dtype=torch.int32, device=dev())
    _same(T.lookup_ewa(uv, g, seed=3, taps=taps), T.lookup_ewa(tail, grad, seed=3, query_offset=N - K, taps=small))
    _same(taps, small)

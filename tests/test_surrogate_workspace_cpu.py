"""Workspace of the surrogate's calls: the convolutions' per-sample partial gradients
are part of it only for networks that a kernel forms them for (kernel size 5, stride
2, small enough for shared memory); every other network needs its activations alone.
A workspace for a batch also serves every smaller one."""
import ctypes as C

import pytest

from paper_1812_10375_gb300 import build


@pytest.fixture(scope="module")
def sur():
    build.build()
    from paper_1812_10375_gb300 import surrogate
    return surrogate


def al(n):
    return (n + 63) & ~63


def activations(L0, C1, C2, C3, K, S, NS, H, NOUT, B):
    """Bytes of the layers' values and gradients and of the two loss terms."""
    lens = []
    for _ in range(3):
        L0 = (L0 - K) // S + 1
        lens.append(L0)
    conv = [B * c * n for c, n in zip((C1, C2, C3), lens)]
    h0, h, y = B * (C3 + NS), B * H, B * NOUT
    return 4 * (3 * sum(map(al, conv)) + 2 * al(h0) + 6 * al(h) + 2 * al(y) + al(2))


def workspace(sur, sizes, B):
    return int(sur._lib().hlb_sur_workspace_bytes(C.byref(sur.hlb_sur_config(*sizes)), B))


@pytest.mark.parametrize("sizes", [
    (500, 16, 32, 32, 3, 2, 2, 256, 6), (500, 16, 32, 32, 5, 1, 2, 256, 6),  # another kernel size, another stride
    (500, 16, 512, 512, 5, 2, 2, 256, 6), (4000, 16, 32, 32, 5, 2, 2, 256, 6)])  # too large for shared memory
@pytest.mark.parametrize("B", [1, 256])
def test_networks_by_layers_need_no_partials(sur, sizes, B):
    assert workspace(sur, sizes, B) == activations(*sizes, B)


@pytest.mark.parametrize("sizes", [
    (1636177817, 1, 1, 1, 5, 2, 1, 8, 2), (858993259, 2, 2, 8, 5, 2, 1, 8, 2), (572662106, 4, 4, 4, 5, 2, 1, 8, 2),
    (409044304, 1, 1, 64, 5, 2, 1, 8, 2)])
def test_layers_beyond_32_bits_do_not_fit_shared_memory(sur, sizes):
    """Sizes of 2^32 floats and a few more: taken modulo 2^32 they are a few KB."""
    assert workspace(sur, sizes, 1) == activations(*sizes, 1)


def test_networks_by_samples_have_their_partials(sur):
    sizes = (500, 16, 32, 32, 5, 2, 2, 256, 6)
    conv = 16 * 5 + 16 + 32 * 16 * 5 + 32 + 32 * 32 * 5 + 32
    last = 0
    for B in range(1, 300):
        n = workspace(sur, sizes, B)
        assert n >= activations(*sizes, B) + 4 * B * conv and n >= last
        last = n


def with_partials(sizes, B, samples):
    """Workspace bytes for a batch of B with partial gradients of `samples` samples."""
    L0, C1, C2, C3, K, S, NS, H, NOUT = sizes
    conv = C1 * K + C1 + C2 * C1 * K + C2 + C3 * C2 * K + C3
    return activations(*sizes, B) + (4 * (al(2 * samples) - al(2) + al(samples * conv)) if samples else 0)


@pytest.mark.parametrize("sizes,batches", [
    # wide linear layers: by layers, but for large batches behind long convolutions
    ((500, 16, 32, 32, 5, 2, 3, 1024, 6), {1: 1, 256: 256, 4096: 4096}),
    ((500, 16, 32, 32, 5, 2, 3, 1280, 6), {1: 0, 255: 0, 256: 256, 4096: 4096}),
    ((500, 16, 32, 32, 5, 2, 3, 2048, 6), {1: 0, 255: 0, 256: 256, 4096: 4096}),
    ((500, 16, 32, 32, 5, 2, 3, 3072, 6), {1: 0, 256: 0, 4096: 0}),
    ((100, 16, 32, 32, 5, 2, 3, 1280, 6), {1: 0, 256: 0, 4096: 0}),
    # short convolutions, not so narrow: by layers from 513 samples on, whose workspace serves 512
    ((64, 4, 8, 8, 5, 2, 3, 768, 6), {512: 512, 513: 512, 4096: 512}),
    ((64, 4, 8, 8, 5, 2, 3, 256, 6), {512: 512, 513: 513, 4096: 4096}),
    ((100, 16, 32, 32, 5, 2, 3, 256, 6), {512: 512, 513: 513, 4096: 4096}),
    # rows that are not whole 16-byte pieces: narrow layers only
    ((500, 16, 32, 32, 5, 2, 3, 255, 6), {1: 1, 256: 256}), ((500, 16, 32, 32, 5, 2, 3, 510, 6), {1: 0, 256: 0}),
    ((500, 16, 32, 33, 5, 2, 3, 512, 6), {1: 0, 256: 0}), ((500, 16, 32, 32, 5, 2, 3, 512, 6), {1: 1, 256: 256})])
def test_which_batches_run_by_samples(sur, sizes, batches):
    for B, samples in batches.items():
        assert workspace(sur, sizes, B) == with_partials(sizes, B, samples), B


def test_workspace_grows_with_the_batch(sur):
    for sizes in [(64, 4, 8, 8, 5, 2, 3, 768, 6), (29, 1, 1, 1, 5, 2, 1, 8, 2), (500, 16, 32, 32, 5, 2, 3, 2048, 6)]:
        n = [workspace(sur, sizes, B) for B in range(1, 4097)]
        assert n == sorted(n)

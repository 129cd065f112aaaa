"""GPU permutation kernel (the transposition of TTGT) against numpy.transpose on an iota payload:
index maps must agree bit for bit."""
import numpy as np
import pytest

from oracle import perm as operm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_2507_20667_gb300 import tnsa
    ctx = tnsa.tn_ctx_create(0, stream=torch.cuda.current_stream().cuda_stream)
    return torch, tnsa, ctx


CASES = [
    ((2,) * 10, None), ((2,) * 20, None), ((3, 5, 7, 2), None), ((33, 65, 3), None),
    ((1, 7, 1, 9), None), ((1000, 1000), (1, 0)), ((4, 4, 4, 4, 4, 4), None), ((17,), (0,)),
    ((2,) * 24, None), ((6, 1, 8, 31, 2), None),
    # the innermost axis survives: rows copied whole (16-byte vectors when aligned, and short rows)
    ((8, 16, 64), (1, 0, 2)), ((2,) * 12, (3, 1, 0, 2, 4, 5, 6, 7, 8, 9, 10, 11)), ((5, 7, 3), (1, 0, 2)),
    ((4, 6, 10), (1, 0, 2)), ((3, 3, 5), (0, 1, 2)),
]


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("elem", [4, 8, 16])
def test_permute_iota_bit_exact(env, case, elem):
    torch, tnsa, ctx = env
    dims, perm = CASES[case]
    rng = np.random.default_rng(case * 10 + elem)
    if perm is None:
        perm = tuple(int(p) for p in rng.permutation(len(dims)))
    n = int(np.prod(dims))
    want = operm.permute_iota(dims, perm, dtype=np.uint32)
    # payload: element i holds iota value i in its first 4 bytes, a fingerprint in the rest
    words = elem // 4
    src = np.zeros((n, words), np.int32)
    src[:, 0] = np.arange(n, dtype=np.int64).astype(np.int32)
    for w in range(1, words):
        src[:, w] = (np.arange(n, dtype=np.int64) * (w + 7) + 3).astype(np.int32)
    d_in = torch.from_numpy(src).cuda()
    d_out = torch.full_like(d_in, -1)
    tnsa.tn_permute(ctx, d_in.data_ptr(), d_out.data_ptr(), elem, dims, perm)
    torch.cuda.synchronize()
    out = d_out.cpu().numpy()
    assert np.array_equal(out[:, 0].astype(np.uint32), want)
    for w in range(1, words):
        assert np.array_equal(out[:, w], src[want.astype(np.int64), w])


def test_permute_rejects_bad_perm(env):
    torch, tnsa, ctx = env
    x = torch.zeros(8, dtype=torch.int64, device="cuda")
    with pytest.raises(tnsa.TnError):
        tnsa.tn_permute(ctx, x.data_ptr(), x.data_ptr(), 8, (2, 4), (0, 0))


# edges of the tiles: chunks cut short in every group, groups that block each other, a surviving run
# that widens the element, one longer than a tile, buffers too badly aligned to widen, more tiles than one
# block takes
EDGE_CASES = [
    ((31, 33, 2), (2, 1, 0), 0), ((129, 3, 61, 5), (3, 1, 0, 2), 0), ((700, 2, 2), (0, 2, 1), 0),
    ((900, 3, 5), (0, 2, 1), 0), ((3, 4097), (1, 0), 0), ((4097, 3), (1, 0), 0), ((5, 3, 2), (1, 0, 2), 0),
    ((5, 3, 6), (1, 0, 2), 1), ((3, 2, 5003), (1, 0, 2), 0), ((2,) * 18, tuple(range(17, -1, -1)), 1),
    ((2,) * 21, tuple(range(14, -1, -1)) + (15, 16, 17, 18, 19, 20), 0), ((300, 300, 40), (2, 1, 0), 0), ((1, 1), (1, 0), 0),
]


@pytest.mark.parametrize("case", range(len(EDGE_CASES)))
@pytest.mark.parametrize("elem", [1, 2, 4, 8, 16])
def test_permute_tile_edges(env, case, elem):
    torch, tnsa, ctx = env
    dims, perm, shift = EDGE_CASES[case]   # shift: elements by which the buffers miss their alignment
    n = int(np.prod(dims))
    src = np.random.default_rng(case).integers(0, 256, (n + shift) * elem, dtype=np.uint8)
    want = src[shift * elem:].reshape(*dims, elem).transpose(*perm, len(dims)).reshape(-1)
    d_in = torch.from_numpy(src).cuda()
    d_out = torch.zeros((n + 2 * shift) * elem, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    tnsa.tn_permute(ctx, d_in.data_ptr() + shift * elem, d_out.data_ptr() + shift * elem, elem, dims, perm)
    tnsa.tn_ctx_synchronize(ctx)
    got = d_out.cpu().numpy()
    assert np.array_equal(got[shift * elem:(n + shift) * elem], want)
    assert not got[:shift * elem].any() and not got[(n + shift) * elem:].any()


# paths chosen by size: tiles whose input axes lie partly in the output's group, whole or about to be cut; long
# surviving runs copied run by run (8, 16 and 32 lanes a run, runs cut into chunks, one run too few);
# transpositions of two long axes (with and without other axes, tiles just over and under half full)
PATH_CASES = [
    ((2,) * 14, (4, 7, 0, 9, 13, 3, 11, 1, 8, 5, 2, 6, 10, 12)), ((3, 2, 5, 7, 2, 3), (4, 2, 0, 3, 5, 1)), ((37, 33, 3, 20, 5), (0, 2, 3, 4, 1)),
    ((2, 1) * 16, tuple(range(31, -1, -1))),
    ((45, 46, 33), (1, 0, 2)), ((64, 33, 65), (1, 0, 2)), ((13, 17, 11, 131), (2, 0, 1, 3)), ((33, 32, 2049), (1, 0, 2)),
    ((23, 89, 33), (1, 0, 2)),
    ((97, 65), (1, 0)), ((129, 3, 63), (2, 1, 0)), ((64, 127), (1, 0)), ((32, 31, 95), (2, 0, 1)), ((1500, 1401), (1, 0)),
    ((33, 700), (1, 0)), ((33, 33), (1, 0)), ((17, 5, 64), (2, 1, 0)),
]


@pytest.mark.parametrize("case", range(len(PATH_CASES)))
@pytest.mark.parametrize("elem", [1, 2, 4, 8, 16])
def test_permute_paths_by_size(env, case, elem):
    torch, tnsa, ctx = env
    dims, perm = PATH_CASES[case]
    n = int(np.prod(dims))
    src = np.random.default_rng(case).integers(0, 256, n * elem, dtype=np.uint8)
    d_in = torch.from_numpy(src).cuda()
    d_out = torch.zeros((n + 2) * elem, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    tnsa.tn_permute(ctx, d_in.data_ptr(), d_out.data_ptr() + elem * (elem < 16), elem, dims, perm)
    tnsa.tn_ctx_synchronize(ctx)
    got = d_out.cpu().numpy()[elem * (elem < 16):]
    want = src.reshape(*dims, elem).transpose(*perm, len(dims)).reshape(-1)
    assert np.array_equal(got[:n * elem], want) and not got[n * elem:].any()


# more than 2^31 - 1 elements that cannot be widened: 64-bit offsets in the tiles and in the runs
@pytest.mark.parametrize("dims,perm", [((46349, 46337), (1, 0)), ((1291, 1301, 1307), (2, 1, 0)), ((1291, 1301, 1307), (1, 0, 2)),
                                       ((130127, 1273, 13), (1, 0, 2))])
def test_permute_more_elements_than_32_bits(env, dims, perm):
    torch, tnsa, ctx = env
    x = torch.randint(0, 256, dims, dtype=torch.uint8, device="cuda")
    out = torch.zeros(x.numel(), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    tnsa.tn_permute(ctx, x.data_ptr(), out.data_ptr(), 1, dims, perm)
    tnsa.tn_ctx_synchronize(ctx)
    assert torch.equal(out.view([dims[p] for p in perm]), x.permute(*perm))

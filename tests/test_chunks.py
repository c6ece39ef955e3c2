"""The planning of the weight gradients on the host: into how many chunks of rows a layer's gradient is cut.  The tensor cores
truncate when they accumulate, so no other need of a call may make the chunks longer: they are held to the number that follows
from the part and the layer alone, restated here."""
import pytest

from paper_2305_09887_b200 import binding, build


@pytest.fixture(scope="module", autouse=True)
def library():
    build.build_library()


def _ceil(a, b):
    return -(-a // b)


def _aligned(n):
    return _ceil(n, 64) * 64


def _fewest(n, parts, blocks):
    """The least number of chunks, of 1,024 rows or more and at most 64, at which waves of blocks on 148 SMs x rows per chunk is within
    3 % of its least; as chunks of whole 64 rows."""
    most = min(64, max(1, _ceil(n, 1024)))

    def cost(ns):
        rows = _aligned(_ceil(n, ns))
        return _ceil(parts * _ceil(n, rows) * blocks, 148) * rows

    best = min(cost(ns) for ns in range(1, most + 1))
    ns = next(ns for ns in range(1, most + 1) if ns == most or cost(ns) <= best * 1.03)
    return _ceil(n, _aligned(_ceil(n, ns)))


def _blocks(nsrc, d_in, d_out):
    """Blocks that work on a chunk, each on up to 256 of the sources' columns and 256 of the gradient's."""
    return _ceil(nsrc * _ceil(d_in, 128), 2) * _ceil(d_out, 256)


def _check(dims, n, parts=1, ddims=None, gemm_dtype=0, variant=(0, 0, 0)):
    got = binding.selftest_chunks(dims, n, parts, ddims, gemm_dtype, variant)
    nsrc = 1 if variant[0] else 2
    for l in range(len(dims) - 1):
        assert got[l] >= min(_fewest(n, parts, _blocks(nsrc, dims[l], dims[l + 1])), _fewest(n, parts, _blocks(1, dims[l], dims[l + 1]))), (l, got)
    if ddims:
        assert got[-1] >= min(_fewest(n, parts, _blocks(1, a, b)) for a, b in zip(ddims[:-1], ddims[1:])), got


@pytest.mark.parametrize("dims, n", [((8, 8, 4), 500_000), ((8, 8, 4), 1_000_000), ((16, 16, 8), 1_000_000), ((16, 16, 8), 5_000_000), ((32, 32, 8), 5_000_000),
                                     ((16, 256, 4), 5_000_000), ((100, 64, 64, 8), 121_000), ((16, 256, 256, 48), 2_000_000)])
@pytest.mark.parametrize("variant", [(0, 0, 0), (0, 1, 1), (1, 0, 0)])
def test_chunks_of_networks_that_are_small_beside_their_part(dims, n, variant):
    _check(dims, n, 1, variant=variant)
    _check(dims, n // 5, 5, variant=variant)


# widths that are no multiple of four: the rows of the partial sums are padded, the scratch counts them unpadded
@pytest.mark.parametrize("dims, n, ddims", [((16, 16, 5), 1_000_000, None), ((16, 16, 5), 4_000_000, None), ((32, 32, 7), 5_000_000, None), ((64, 90, 3), 1_000_000, None),
                                            ((10, 33, 3), 200_000, None), ((8, 5), 1_000_000, None), ((64, 256, 256), 131_072, (256, 1)), ((64, 128, 128), 1_000_000, (128, 1)),
                                            ((64, 64, 30), 500_000, (30, 7, 1))])
def test_chunks_of_widths_whose_partial_sums_are_padded(dims, n, ddims):
    _check(dims, n, 1, ddims)
    _check(dims, n // 3, 3, ddims)


# layers whose sources are wider than what a block takes: however a chunk is cut into blocks, it is no longer for it
@pytest.mark.parametrize("dims, n, parts", [((512, 64), 13_800, 16), ((512, 128), 9_700, 16), ((512, 96), 57_600, 16), ((512, 128), 10_072, 23), ((1024, 128), 3_152, 23),
                                            ((512, 90), 7_991, 64), ((512, 512), 62_500, 8), ((128, 256, 256), 25_000, 8)])
@pytest.mark.parametrize("gemm_dtype", [0, 1])
def test_chunks_of_wide_layers(dims, n, parts, gemm_dtype):
    got = binding.selftest_chunks(dims, n, parts, gemm_dtype=gemm_dtype)
    for chunks, a, b in zip(got, dims[:-1], dims[1:]):
        assert chunks >= _fewest(n, parts, _blocks(2, a, b)), (a, b, got)

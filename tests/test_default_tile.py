"""The tile that a product takes by default, where narrow and wide ones were
measured far apart (host only: no GPU needed)."""
import pytest


@pytest.mark.parametrize("prec,M,K,N,tile", [
    # one wave of pairs, two of 128 x 128 under half of the masks
    ("bf16", 2048, 8192, 1024, 256), ("bf16x3", 2048, 8192, 1024, 256), ("fp16x3", 2048, 8192, 1024, 256),
    ("fp32", 2048, 8192, 1024, 256), ("bf16x3", 4096, 6144, 512, 256), ("bf16", 1000, 4096, 2048, 256),
    # several waves
    ("bf16x3", 8192, 8192, 8192, 256), ("fp32", 8192, 8192, 8192, 256), ("bf16", 8192, 8192, 8192, 256),
    # few tiles
    ("bf16x3", 512, 256, 128, 64), ("fp16x3", 1000, 1416, 1100, 128), ("fp32", 1000, 1024, 1024, 128),
    ("fp32", 512, 256, 128, 0), ("exact", 512, 256, 128, 256)])
def test_default_tile(libbpx, prec, M, K, N, tile):
    code = libbpx.Code.systematic(8, 3, 8)
    assert libbpx.default_tile(code, libbpx.PRECISIONS[prec], N, K, -(-M // code.num_sources)) == tile


def test_refused(libbpx):
    code = libbpx.Code.table1()
    for prec, N, K, h in ((99, 128, 128, 4), (0, 127, 128, 4), (0, 128, 127, 4), (0, 128, 128, 0)):
        with pytest.raises(libbpx.BpxError) as err:
            libbpx.default_tile(code, prec, N, K, h)
        assert err.value.code == libbpx.ERR_INVAL

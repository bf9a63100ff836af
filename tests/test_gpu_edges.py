"""Sizes at the edges of the kernels' tiles and of the rules that choose between them, against the oracle."""
import pytest

import workloads as wl
from test_gpu_kernels import TOL_TENSOR, _conv_case
from test_gpu_step import check_step

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,ks,st,ci,co,H", [
    (1, 3, 1, 16, 16, 1),        # a map of one pixel: the block is mostly padding
    (3, 3, 1, 32, 16, 5),        # whole maps per copy (6 x 6 padded positions); ragged last tile
    (2, 3, 1, 16, 48, 6),        # 7 x 7 = 49 positions: one copy per row; a column group of 16
    (1, 3, 1, 16, 16, 252),      # a wide map without column strips
    (1, 3, 1, 16, 16, 255),      # the narrowest with them
    (2, 3, 1, 512, 512, 2),      # few positions, a long K loop: split over CTAs
    (9, 1, 1, 64, 80, 3),        # 81 pixels: less than a tile
    (5, 1, 1, 16, 256, 32),      # two channel slices; weights resident
    (2, 1, 1, 512, 256, 8),      # exactly one tile; the weight ring
    (7, 1, 2, 32, 64, 7),        # odd map, strided: zeros between the samples up to the border
    (2, 1, 2, 48, 32, 10),
    (13, 3, 1, 128, 128, 14)], ids=str)
@pytest.mark.parametrize("path", [0, 2])
def test_convolutions_at_the_edges_of_the_tiling(N, ks, st, ci, co, H, path):
    e = _conv_case(ks, st, ci, co, H, N, path)
    assert max(e) <= (2e-5 if path == 0 else TOL_TENSOR), e


@pytest.mark.parametrize("N,ks,st,ci,co,H", [
    (37, 1, 1, 32, 16, 32),      # 296 tiles: the most the tile kernel takes; its data gradient is as wide as it may be
    (38, 1, 1, 32, 16, 32),      # 304: pipelined
    (37, 1, 1, 48, 64, 16),      # 74 tiles of 64 channels, 48 the other way
    (75, 1, 1, 16, 256, 16),     # pipelined forward, the tile kernel's data gradient
    (75, 1, 1, 96, 96, 16),      # one pass on the tile kernel, three pipelined
    (37, 1, 2, 64, 48, 15),      # strided, ragged tiles: the data gradient beyond its quarter of the line
    (2, 1, 2, 16, 32, 9)], ids=str)
@pytest.mark.parametrize("path", [0, 2])
def test_one_by_one_windows_on_either_side_of_the_kernels_line(N, ks, st, ci, co, H, path):
    e = _conv_case(ks, st, ci, co, H, N, path)
    assert max(e) <= (2e-5 if path == 0 else TOL_TENSOR), e


@pytest.mark.parametrize("N,ks,st,ci,co,H", [
    (1, 3, 1, 3, 16, 5),         # a stem: 16-wide tiles, the k steps shared by the block's warps
    (3, 7, 2, 3, 64, 17),
    (2, 3, 2, 16, 32, 9),        # strided: four classes of input positions of unequal size
    (2, 3, 2, 24, 17, 8),
    (1, 1, 2, 5, 33, 7),         # classes without a tap receive zeros
    (4, 1, 1, 7, 65, 3)], ids=str)
def test_cuda_core_convolutions_at_the_edges_of_the_tiling(N, ks, st, ci, co, H):
    e = _conv_case(ks, st, ci, co, H, N, 1)
    assert max(e) <= 2e-5, e


@pytest.mark.parametrize("ksize,size", [(2, 9), (2, 8), (3, 17), (3, 2)])
def test_max_pools_on_odd_maps_and_a_head_wider_than_its_blocks(ksize, size):
    """A pool whose input also feeds nothing else, on odd and even maps; 260 channels and 11 classes leave the head's blocks
    of 256 channels and 8 classes ragged."""
    ops = [wl.Op(wl.CONV, -1, -1, 3, 16, 3, 1, 1, 0.0), wl.Op(wl.MAXPOOL, 0, -1, 16, 16, ksize, 2, ksize // 3, 0.0),
           wl.Op(wl.CONV, 1, -1, 16, 260, 1, 1, 0, 0.0), wl.Op(wl.HEAD, 2, -1, 260, 11, 0, 1, 0, 0.0)]
    check_step(ops, (size, size, 3), 6, 3, [2], seed=21)


@pytest.mark.parametrize("batch", [30, 33])
def test_batch_norm_backward_from_the_sums_of_the_data_gradient(batch):
    """Tensors of a BN too large for one launch of clusters: the data gradients form the sums (1x1 and 3x3, 64 and 16
    channels), the shortcut adds on the way; ragged last tiles."""
    ops = wl.resnet_v2_cifar(1, widths=(64,), outs=(64,))
    check_step(ops, (33, 33, 3), batch, 1, [5], seed=22, bn_jitter=0.2)

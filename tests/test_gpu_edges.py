"""Sizes at the edges of the kernels' tiles and of the rules that choose between them, against the oracle."""
import numpy as np
import pytest
import torch

import paper_1911_05146_b200 as hpf
import workloads as wl
from test_gpu_kernels import TOL_TENSOR, _conv_case
from hpf_testlib import Bound, seeded
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


@pytest.mark.parametrize("N,ks,st,ci,co,H", [
    (75, 1, 1, 16, 256, 16),     # two slices of 128 channels, each of a lane's eight in two pieces of four
    (38, 1, 1, 32, 16, 32),      # 16 channels forward, 32 the other way
    (3, 3, 1, 64, 96, 9),        # padded grid, three groups of 32 channels
    (2, 3, 1, 512, 512, 2),      # split over CTAs
    (5, 1, 2, 64, 64, 15)], ids=str)      # zeros between the samples
@pytest.mark.parametrize("path", [0, 2])
def test_results_that_start_at_any_sixteen_bytes(N, ks, st, ci, co, H, path):
    """The write-out stores 32 bytes a lane where the buffer allows it and 16 otherwise: the same bits."""
    P, dev = (H - 1) // st + 1, "cuda:0"
    g = torch.Generator(device=dev)
    g.manual_seed(N)
    x, dy = torch.randn(N, H, H, ci, generator=g, device=dev), torch.randn(N, P, P, co, generator=g, device=dev)
    w = torch.randn(co, ks, ks, ci, generator=g, device=dev) * (2.0 / (ci * ks * ks)) ** 0.5
    args = (N, H, H, ci, co, ks, st, ks // 2, path)
    wprep, scratch = torch.empty(4 * w.numel(), device=dev), torch.zeros(hpf.conv_scratch_bytes(*args[:8]), dtype=torch.uint8, device=dev)
    hpf.conv_prepare_weights(w, wprep, ci, co, ks)
    out = []
    for skip in (0, 4):
        y, dx = (torch.full((t.numel() + 4,), float("nan"), device=dev)[skip:skip + t.numel()] for t in (dy, x))
        hpf.conv_fwd(x, w, wprep, y, *args, scratch)
        hpf.conv_dgrad(dy, w, wprep, dx, *args, scratch)
        out.append((y, dx))
    torch.cuda.synchronize()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert not torch.isnan(out[1][0]).any() and not torch.isnan(out[1][1]).any()


@pytest.mark.parametrize("C,ks,size", [(48, 3, 9), (64, 1, 7), (1040, 1, 3)], ids=str)      # a lane's channels change from row to row; stay; more than a block's threads
@pytest.mark.parametrize("cuts", [[], [2], [3], [4]], ids=str)
def test_a_plain_batch_norm_ends_its_block(C, ks, size, cuts):
    """BN, residual sum and ReLU in one launch, as far as they stand in one partition."""
    ops = [wl.Op(wl.CONV, -1, -1, 3, C, 3, 1, 1, 0.0), wl.Op(wl.CONV, 0, -1, C, C, ks, 1, ks // 2, 0.0), wl.Op(wl.BN, 1, -1, C, C, 0, 1, 0, 1e-5),
           wl.Op(wl.ADD, 2, 0, C, C, 0, 1, 0, 0.0), wl.Op(wl.RELU, 3, -1, C, C, 0, 1, 0, 0.0), wl.Op(wl.HEAD, 4, -1, C, 10, 0, 1, 0, 0.0)]
    check_step(ops, (size, size, 3), 6, 3, cuts, seed=23, bn_jitter=0.2)


def test_a_plain_batch_norm_and_its_sum_without_an_activation():
    """(No BN may follow the sum: it would remove what the first one's shift adds, whose gradient would be zero plus rounding.)"""
    ops = [wl.Op(wl.CONV, -1, -1, 3, 32, 3, 1, 1, 0.0), wl.Op(wl.CONV, 0, -1, 32, 32, 3, 1, 1, 0.0), wl.Op(wl.BN, 1, -1, 32, 32, 0, 1, 0, 1e-5),
           wl.Op(wl.ADD, 0, 2, 32, 32, 0, 1, 0, 0.0), wl.Op(wl.HEAD, 3, -1, 32, 10, 0, 1, 0, 0.0)]
    check_step(ops, (8, 8, 3), 4, 2, [], seed=24, bn_jitter=0.2)


@pytest.mark.parametrize("kind", [wl.BN, wl.BNRELU], ids=["BN", "BNRELU"])
@pytest.mark.parametrize("C", [4096, 4224, 24576, 24704])      # 48 KB of shared memory and the next; the most channels that fit and the next
def test_a_batch_norm_of_very_many_channels_behind_a_convolution(C, kind):
    ops = [wl.Op(wl.CONV, -1, -1, 3, 16, 3, 1, 1, 0.0), wl.Op(wl.CONV, 0, -1, 16, C, 1, 1, 0, 0.0), wl.Op(kind, 1, -1, C, C, 0, 1, 0, 1e-5),
           wl.Op(wl.CONV, 2, -1, C, 16, 1, 1, 0, 0.0), wl.Op(wl.HEAD, 3, -1, 16, 10, 0, 1, 0, 0.0)]
    check_step(ops, (4, 4, 3), 4, 2, [], seed=25, bn_jitter=0.2)


@pytest.mark.parametrize("C,ks,size,batch,micro,shift", [(64, 1, 8, 8, 2, 0), (64, 3, 8, 4, 1, 0), (256, 1, 9, 5, 1, 0), (16, 3, 32, 16, 2, 30)], ids=str)
def test_statistics_of_a_plain_batch_norm_behind_a_convolution(C, ks, size, batch, micro, shift):
    """Mean and 1/sigma as fp64 statistics of the stored values give them.  y = (x - mean) / sigma is a straight line in x, so
    both come out of a fit far more precisely than one value of y has them.  The mean is off by its own rounding and the fp32 sums
    of a lane's few rows, values of about sigma: together less than 2^-24 sigma.  1/sigma: its own rounding, half a unit in the
    last place, and half the relative error of the sum of squares, some 2^-24: less than 1.25 units."""
    ops = [wl.Op(wl.CONV, -1, -1, 3, 16, 3, 1, 1, 0.0), wl.Op(wl.CONV, 0, -1, 16, C, ks, 1, ks // 2, 0.0), wl.Op(wl.BN, 1, -1, C, C, 0, 1, 0, 1e-5),
           wl.Op(wl.HEAD, 2, -1, C, 10, 0, 1, 0, 0.0)]
    x, labels, theta = seeded(ops, (size, size, 3), batch, 31)
    bd = Bound(ops, (size, size, 3), batch, micro, [], theta)
    bd.upload(x + np.float32(shift), labels)
    bd.step()
    for m in range(micro):
        v, y = (bd.tensor(i, m).astype(np.float64).reshape(-1, C) for i in (1, 2))
        mean, sigma = v.mean(0), np.sqrt(v.var(0) + 1e-5)
        slope = ((v - mean) * (y - y.mean(0))).sum(0) / ((v - mean) ** 2).sum(0)
        used_mean = mean - y.mean(0) / slope
        ulp = lambda a: np.spacing(np.abs(a).astype(np.float32)).astype(np.float64)  # noqa: E731
        assert (np.abs(used_mean - mean) <= 0.5 * ulp(mean) + 2.0 ** -24 * sigma).all(), (np.abs(used_mean - mean) / sigma).max()
        assert (np.abs(slope - 1.0 / sigma) <= 1.25 * ulp(1.0 / sigma)).all(), (np.abs(slope - 1.0 / sigma) / ulp(1.0 / sigma)).max()


def test_when_launches_trigger_their_successors_changes_no_bit():
    """Every forward convolution late (the default), those of cells that run beside another one, and none."""
    ops = wl.resnet_v2_cifar(1)
    x, labels, theta = seeded(ops, (32, 32, 3), 8, 32)
    out = []
    for options in ({}, {hpf.OPT_PDL_LATE_FROM: 2}, {hpf.OPT_PDL_LATE_FROM: 1000}, {hpf.OPT_PDL: 0}):
        bd = Bound(ops, (32, 32, 3), 8, 2, [9], theta, options, backward_streams=True)
        bd.upload(x, labels)
        out.append((bd.step(one_graph=True), bd.slots.cpu().numpy()))
    for loss, slots in out[1:]:
        assert loss == out[0][0] and np.array_equal(slots, out[0][1])


def test_persistent_cells_form_a_plain_batch_norms_moments_like_single_launches():
    """(In a cell the fp64 sums are a branch of the write-out, alone a kernel of their own.)"""
    c = wl.config("r8v1")
    x, labels, theta = seeded(c["ops"], c["in_hwc"], c["B"], 33, 0.2)
    out = []
    for ctas in (0, 16):
        bd = Bound(c["ops"], c["in_hwc"], c["B"], c["M"], c["cuts"], theta, {hpf.OPT_CELL_CTAS: ctas, hpf.OPT_GROUP_LAUNCHES: 0})
        bd.upload(x, labels)
        out.append((bd.step(), bd.slots.cpu().numpy(), bd.model.launch_count()))
    assert out[1][2] < out[0][2] and out[0][0] == out[1][0] and np.array_equal(out[0][1], out[1][1])

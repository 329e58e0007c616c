"""Row-tile passes, readout pass and coil-numbered one-pass kernel at the sizes where their tilings can go wrong, against
the CPU oracle: forward, VJP and A^H y of the same inputs."""
import numpy as np
import pytest

from oracle.oracle import MASK_FULL, MASK_READOUT_INVARIANT
from tests.gpu_common import assert_close, run_gpu
from tests.test_gpu_parity import problem

pytestmark = pytest.mark.gpu


def check_all(oracle, d, x, y, sens, mask, eta, what):
    import torch
    import paper_2207_08393_b200 as g
    for yy, ref, name in ((y, oracle.dc_forward(x, y, sens, mask, eta, d, nthreads=8), "forward"),
                          (None, oracle.dc_vjp(x, sens, mask, eta, d, nthreads=8), "vjp")):
        got = run_gpu(x, yy, sens, mask, eta, d.fft_rank, d.sens_has_frames, d.mask_kind)
        assert_close(got, ref, x, what + " " + name)
    zero = np.zeros_like(x)
    ref = oracle.dc_forward(zero, y, sens, mask, 1.0, d, nthreads=8)      # 0 - (A^H (A 0 - y))
    dc = g.DataConsistency(d.batch, d.coils, d.frames, d.fft_rank, d.n, d.sens_has_frames, d.mask_kind)
    dev = torch.device("cuda:0")
    out = dc.adjoint(*(torch.from_numpy(a).to(dev) for a in (y, sens, mask)))
    torch.cuda.synchronize()
    assert_close(out.cpu().numpy(), ref, ref, what + " adjoint")


# n1: rows per block and middle radix (1 x 20, 2 x 23, 12 x 32, 16 x 32, 20 x 32); n2: columns per block (single-stage
# rows, a last warp with 8 or 14 idle lanes, both stage buffers, one buffer for both, the largest tile)
@pytest.mark.parametrize("n", [(1, 20, 16), (1, 46, 40), (1, 384, 46), (1, 512, 24), (1, 640, 32), (1, 320, 368), (1, 40, 640), (1, 16, 512)])
@pytest.mark.parametrize("coils", [1, 5])
def test_slices_with_an_arbitrary_mask(oracle, n, coils):
    d, x, y, sens, mask = problem(2, 1, coils, 1, n, MASK_FULL, weighted=(coils == 5), seed=sum(n), density=0.3)
    check_all(oracle, d, x, y, sens, mask, 0.9, "slice %s" % (n,))


# z values of a ky group in the middle pass: every group larger than the 2048 that are staged, groups on both sides of it, a full
# mask, groups of a few samples and of none
@pytest.mark.parametrize("n,density", [((2, 368, 320), 0.3), ((2, 368, 320), 0.2785), ((2, 320, 96), 1.0), ((2, 64, 40), 0.02), ((4, 160, 24), 0.003)])
def test_groups_of_z_values(oracle, n, density):
    import torch
    import paper_2207_08393_b200 as g
    d, x, y, sens, mask = problem(3, 1, 2, 1, n, MASK_READOUT_INVARIANT, weighted=False, seed=sum(n), density=density)
    mask = (mask * np.random.default_rng(1).uniform(0.5, 1.5, mask.shape)).astype(np.float32)
    check_all(oracle, d, x, y, sens, mask, 0.9, "groups %s" % (n,))
    dc = g.DataConsistency(1, 2, 1, 3, n)
    t = [torch.from_numpy(a).to("cuda:0") for a in (x, y, sens, mask)]
    dc.prepare(t[1], t[3])
    assert torch.equal(dc.forward_prepared(t[0], t[1], t[2], t[3], 0.9), g.DataConsistency(1, 2, 1, 3, n).forward(t[0], t[1], t[2], t[3], 0.9))


# 23-point rows: outputs stored as they are formed (long rows) or after the butterfly, few and many rows a block
@pytest.mark.parametrize("n", [(4, 92, 184), (2, 46, 368), (6, 20, 184), (2, 92, 92), (2, 64, 184), (2, 92, 46), (2, 240, 184), (1, 92, 368), (1, 6, 184)])
def test_rows_of_23_points(oracle, n):
    rank = 3 if n[0] > 1 else 2
    for kind in (MASK_READOUT_INVARIANT, MASK_FULL) if rank == 3 else (MASK_FULL,):
        d, x, y, sens, mask = problem(rank, 1, 3, 1, n, kind, seed=sum(n), density=0.3)
        check_all(oracle, d, x, y, sens, mask, 0.9, "rows of 23 points %s" % (n,))


# blocks of passes 1 and 3 that are resident on an SM (their registers decide), per pass; 24-point rows keep their twiddles in registers
# (fewer blocks) unless the others save a round
@pytest.mark.parametrize("n,fwd,inv,loose", [((24, 80, 46), 10, 8, False), ((24, 92, 92), 6, 6, False), ((368, 64, 24), 20, 20, False), ((24, 64, 24), 20, 16, True)])
def test_resident_blocks_of_the_row_tile_passes(n, fwd, inv, loose):
    import torch
    import paper_2207_08393_b200 as g
    from tests.test_gpu_dispatch import captured
    dev = torch.device("cuda:0")
    x = torch.zeros((1, 1) + n, dtype=torch.complex64, device=dev)
    s = torch.zeros((1, 3) + n, dtype=torch.complex64, device=dev)
    dc, m = g.DataConsistency(1, 3, 1, 3, n), torch.ones((1, 1) + n[1:], device=dev)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    launches = captured(lambda: dc.vjp(x, s, m, 1.0))
    for name, least in (("tile_fwd_kernel", fwd), ("tile_inv_kernel", inv)):
        k, = [k for k in launches if name in k["name"]]
        assert k["resident"] >= least * sms, k
        assert ("Lb1E" in k["name"]) == (loose and "inv" in name), k


# short tiles with 23-point rows: the form with more blocks on an SM only where that saves a round of them
@pytest.mark.parametrize("n,coils,batch", [((32, 46, 184), 3, 1), ((24, 46, 184), 3, 1), ((1, 92, 184), 5, 12), ((1, 46, 368), 3, 6), ((1, 46, 368), 3, 8),
                                           ((48, 92, 184), 2, 1), ((1, 20, 368), 3, 3), ((1, 92, 184), 6, 3)])
def test_form_of_short_tiles(oracle, n, coils, batch):
    import torch
    import paper_2207_08393_b200 as g
    from tests.test_gpu_dispatch import captured
    rank, kind = (3, MASK_READOUT_INVARIANT) if n[0] > 1 else (2, MASK_FULL)
    d, x, y, sens, mask = problem(rank, batch, coils, 1, n, kind, seed=sum(n), density=0.3)
    check_all(oracle, d, x, y, sens, mask, 0.9, "short tiles %s" % (n,))
    dc = g.DataConsistency(batch, coils, 1, rank, n, 0, kind)
    t = [torch.from_numpy(a).to("cuda:0") for a in (x, sens, mask)]
    launches = captured(lambda: dc.vjp(t[0], t[1], t[2], 1.0))
    for name in ("tile_fwd_kernel", "tile_inv_kernel"):
        k, = [k for k in launches if name in k["name"]]
        rounds = lambda per_sm: -(-k["blocks"] // (per_sm * torch.cuda.get_device_properties(0).multi_processor_count))
        taken = -(-k["blocks"] // k["resident"])
        # blocks on an SM of the tight form (80 registers), and of the other one at most (92 and more)
        if "Lb1E" in k["name"]:
            assert taken <= rounds(4 if n[2] == 184 else 2), k
        else:
            assert taken < rounds(3 if n[2] == 184 else 1), k


# middle radix 16 with full blocks: weights and measurements take 48 KB of shared memory, the twiddles come on top
@pytest.mark.parametrize("n", [(1, 160, 240), (1, 256, 256), (1, 160, 512)])
def test_slices_whose_middle_pass_takes_48_kb(oracle, n):
    d, x, y, sens, mask = problem(2, 1, 2, 1, n, MASK_FULL, seed=sum(n), density=0.3)
    check_all(oracle, d, x, y, sens, mask, 0.9, "slice %s" % (n,))


# readout pass: columns per block 32 / 16 with a remainder, single-stage and two-stage lengths, radix 32, prime radix
@pytest.mark.parametrize("n", [(4, 12, 46), (20, 6, 20), (46, 8, 24), (96, 4, 40), (128, 6, 10), (160, 4, 16), (512, 2, 12), (640, 2, 20)])
def test_volumes_with_an_arbitrary_mask(oracle, n):
    d, x, y, sens, mask = problem(3, 1, 3, 1, n, MASK_FULL, weighted=(n[0] == 96), seed=sum(n), density=0.3)
    check_all(oracle, d, x, y, sens, mask, 1.0, "volume %s" % (n,))


# bricks of k0 group x readout x columns: every middle radix, 16, 8 and 4 columns with a remainder, prime radices of the readout, the
# largest bricks, batches and frames; and sizes next to them that take three passes: radix 32 of the readout or of ky, bricks that
# do not fit an SM (368 points with radices 20 and 23 of ky)
@pytest.mark.parametrize("B,T,n", [(1, 1, (24, 24, 20)), (2, 2, (46, 40, 24)), (1, 1, (48, 48, 46)), (1, 2, (96, 160, 10)), (1, 1, (92, 46, 12)),
                                   (1, 1, (120, 120, 6)), (1, 1, (40, 192, 40)), (1, 1, (64, 240, 24)), (1, 1, (384, 48, 4)), (1, 1, (368, 128, 2)),
                                   (1, 1, (160, 320, 12)), (1, 1, (184, 320, 2)), (1, 1, (32, 384, 4)), (1, 1, (320, 120, 10)),
                                   (1, 1, (368, 320, 2)), (1, 1, (368, 46, 4))])
def test_bricks_of_volumes_with_an_arbitrary_mask(oracle, B, T, n):
    d, x, y, sens, mask = problem(3, B, 2, T, n, MASK_FULL, weighted=(n[0] == 96), seed=sum(n), density=0.2)
    check_all(oracle, d, x, y, sens, mask, 0.8, "brick %s" % (n,))


# bricks: unsampled measurements are NaN.  Pairs of neighbouring kz are copied where one of them was sampled (last length a multiple
# of 4), else one at a time; 16, 8 and 4 columns, A^H y by the bricks and by its own passes (40 points)
@pytest.mark.parametrize("n", [(96, 160, 12), (46, 40, 24), (40, 48, 20), (48, 48, 46), (96, 96, 10), (184, 320, 4), (128, 64, 40)])
def test_bricks_do_not_use_unsampled_measurements(oracle, n):
    import torch
    import paper_2207_08393_b200 as g
    d, x, y, sens, mask = problem(3, 1, 2, 1, n, MASK_FULL, weighted=True, seed=sum(n))
    mask *= np.random.default_rng(n[0]).uniform(size=mask.shape) < 0.3
    clean = y.copy()
    y[np.broadcast_to(mask[:, None] == 0, y.shape)] = np.nan
    clean[np.isnan(y)] = 0
    got = run_gpu(x, y, sens, mask, 0.8, 3, 0, MASK_FULL)
    assert_close(got, oracle.dc_forward(x, clean, sens, mask, 0.8, d, nthreads=8), x, "brick %s" % (n,))
    dc = g.DataConsistency(1, 2, 1, 3, n, 0, g.GLEAM_MASK_FULL)
    got = dc.adjoint(*(torch.from_numpy(a).to(torch.device("cuda:0")) for a in (y, sens, mask)))
    torch.cuda.synchronize()
    ref = oracle.dc_forward(np.zeros_like(x), clean, sens, mask, 1.0, d, nthreads=8)
    assert_close(got.cpu().numpy(), ref, ref, "brick %s adjoint" % (n,))


# coils dealt to clusters of 1, 2 and 4 blocks (few tiles), with coil counts that do not divide; frames and batches
@pytest.mark.parametrize("B,C,T,n", [(1, 2, 1, (2, 64, 80)), (1, 7, 1, (2, 92, 64)), (2, 4, 2, (2, 24, 128)), (1, 3, 1, (40, 20, 32)), (1, 6, 1, (2, 640, 20))])
def test_coil_split_of_the_row_tiles(oracle, B, C, T, n):
    d, x, y, sens, mask = problem(3, B, C, T, n, MASK_READOUT_INVARIANT, sens_has_frames=int(T > 1), seed=sum(n) + C, density=0.2)
    check_all(oracle, d, x, y, sens, mask, 0.8, "split %s" % (n,))


# one-pass kernel: lines per warp 1 ... 8 with idle lanes, prime radices, lines beyond the end, more samples than are staged
@pytest.mark.parametrize("n2", [46, 92, 184, 368, 384, 512, 640])
@pytest.mark.parametrize("rows,coils,density", [(2, 2, 0.1), (10, 3, 0.9), (20, 16, 0.2)])
def test_one_pass_kernel_of_slices(oracle, n2, rows, coils, density):
    d, x, y, sens, mask = problem(2, 1, coils, 1, (1, rows, n2), MASK_READOUT_INVARIANT, seed=n2 + rows, density=density)
    check_all(oracle, d, x, y, sens, mask, 0.9, "n2=%d rows=%d" % (n2, rows))


# the same: several coils per warp of a block (24, 32 points), masks of one sample and of all of them, more groups of lines
# than one round holds
@pytest.mark.parametrize("B,C,rows,n2,density", [(8, 16, 32, 24, 0.3), (2, 15, 46, 32, 0.02), (1, 7, 10, 32, 1.0), (1, 5, 6, 256, 0.01),
                                                 (2, 3, 20, 256, 1.0), (8, 2, 640, 368, 0.2)])
def test_one_pass_kernel_by_the_number_of_lines(oracle, B, C, rows, n2, density):
    d, x, y, sens, mask = problem(2, B, C, 1, (1, rows, n2), MASK_READOUT_INVARIANT, seed=n2 + C, density=density)
    check_all(oracle, d, x, y, sens, mask, 0.9, "n2=%d rows=%d coils=%d" % (n2, rows, C))


# volumes: no staged samples left over, fewer and more samples per group of middle lines than are staged
@pytest.mark.parametrize("n,density", [((2, 46, 320), 1.0), ((4, 46, 92), 0.5), ((2, 640, 24), 0.01)])
def test_samples_of_the_middle_pass(oracle, n, density):
    d, x, y, sens, mask = problem(3, 1, 3, 1, n, MASK_READOUT_INVARIANT, seed=sum(n), density=density)
    check_all(oracle, d, x, y, sens, mask, 0.7, "middle pass %s" % (n,))


# one-pass kernel with measurements: frames without samples, with few, with more than a quarter and with all of them, whose
# lines share a warp (4, 2 and 1 lines per warp, rows that leave lines past the end), one and several rounds of units,
# one block per SM (18 frames of 120 rows); unsampled measurements are NaN
@pytest.mark.parametrize("n2,rows,C,T", [(32, 10, 3, 5), (48, 6, 2, 5), (80, 2, 3, 5), (96, 6, 3, 4), (128, 10, 3, 5), (160, 120, 3, 18), (184, 6, 3, 4),
                                         (192, 4, 2, 4), (256, 6, 3, 4), (320, 10, 3, 4), (384, 2, 3, 4), (512, 2, 3, 4)])
def test_measurements_of_frames_of_unlike_density(oracle, n2, rows, C, T):
    d, x, y, sens, mask = problem(2, 1, C, T, (1, rows, n2), MASK_READOUT_INVARIANT, seed=n2 + rows, weighted=True)
    rng = np.random.default_rng(n2)
    for t in range(T):
        keep = rng.uniform(size=n2) < (0.0, 0.1, 0.5, 1.0)[t % 4]
        mask[:, t] *= keep
        y[:, :, t][..., ~keep] = np.nan
    clean = np.nan_to_num(y)
    assert_close(run_gpu(x, y, sens, mask, 0.9, 2, 0, MASK_READOUT_INVARIANT), oracle.dc_forward(x, clean, sens, mask, 0.9, d, nthreads=8), x, "n2=%d" % n2)
    import torch
    import paper_2207_08393_b200 as g
    dev = torch.device("cuda:0")
    dc = g.DataConsistency(1, C, T, 2, (1, rows, n2))
    tx, ty, ts, tm = (torch.from_numpy(a).to(dev) for a in (x, y, sens, mask))
    got = dc.adjoint(ty, ts, tm)
    torch.cuda.synchronize()
    ref = oracle.dc_forward(np.zeros_like(x), clean, sens, mask, 1.0, d, nthreads=8)
    assert_close(got.cpu().numpy(), ref, ref, "n2=%d adjoint" % n2)

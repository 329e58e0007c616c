"""GPU parity of the MoDL model inversion (Eq. 7): gleam_modl_cg_forward / gleam_modl_cg_vjp through
the C ABI against the CPU oracle's conjugate-gradient solve, element by element on the same
seeded inputs.

Tolerance: relative L2 <= 2e-5, max abs error <= 1e-4 * max|oracle result| (the bound of the
gradient data-consistency step).  One operator application in single precision deviates by about
1e-7 (relative) from the double-precision one; the conjugate-gradient recurrences amplify
perturbations of their vectors by at most about the condition number of A^H A + mu I
(<= (1 + mu) / mu = 21 for the paper's mu = 0.05 with unit-norm sensitivities), and since the
inner products are accumulated in double precision the steps do not add to it: 21 * 1e-7 = 2e-6
(measured on the full-size workloads: 1.9e-6 after 10 and after 30 steps), a factor 10 of margin.
"""
import numpy as np
import pytest

from oracle.oracle import Dims, MASK_FULL, MASK_READOUT_INVARIANT
from paper_2207_08393_b200 import workloads as wl
from tests.gpu_common import run_gpu_modl
from tests.test_gpu_parity import crandn, workload_case

pytestmark = pytest.mark.gpu

REL_L2_TOL = 2e-5
MAX_ABS_TOL = 1e-4


def close(got, ref, what):
    got = np.asarray(got).astype(np.complex128)
    assert np.isfinite(got.view(np.float64)).all(), what + ": non-finite output"
    scale = max(np.abs(ref).max(), 1e-300)
    rel = np.linalg.norm(got - ref) / max(np.linalg.norm(ref), 1e-300)
    mab = np.abs(got - ref).max() / scale
    assert rel <= REL_L2_TOL, "%s: rel L2 %.3e > %.1e" % (what, rel, REL_L2_TOL)
    assert mab <= MAX_ABS_TOL, "%s: max abs %.3e > %.1e (units of max|result|)" % (what, mab, MAX_ABS_TOL)
    return rel


def problem(rank, B, C, T, n, mask_kind, sens_has_frames=0, weighted=False, seed=0, density=0.4):
    rng = np.random.default_rng(seed)
    d = Dims(B, C, T, rank, tuple(n), sens_has_frames, mask_kind)
    z = crandn(rng, *d.image_shape()); y = crandn(rng, *d.kspace_shape())
    sens = crandn(rng, *d.sens_shape())
    sens = (sens / np.sqrt(np.sum(np.abs(sens) ** 2, axis=1, keepdims=True))).astype(np.complex64)
    if weighted:
        mask = rng.uniform(0, 1, d.mask_shape()).astype(np.float32)
    else:
        mask = (rng.uniform(size=d.mask_shape()) < density).astype(np.float32)
    return d, z, y, sens, mask


def check(oracle, d, z, y, sens, mask, mu, n_iter, what, in_place=False):
    ref = oracle.modl_cg_forward(z, y, sens, mask, mu, n_iter, d, nthreads=8)
    got = run_gpu_modl(z, y, sens, mask, mu, n_iter, d.fft_rank, d.sens_has_frames, d.mask_kind, in_place=in_place)
    close(got, ref, what + " solve")
    refv = oracle.modl_cg_vjp(z, sens, mask, mu, n_iter, d, nthreads=8)
    gotv = run_gpu_modl(z, None, sens, mask, mu, n_iter, d.fft_rank, d.sens_has_frames, d.mask_kind, in_place=in_place)
    close(gotv, refv, what + " vjp")


@pytest.mark.parametrize("n_iter", [1, 2, 3, 10])
@pytest.mark.parametrize("mu", [0.05, 4.0])            # the paper's values for R = 16 and R = 4
def test_rank2_steps_and_mu(oracle, n_iter, mu):
    d, z, y, sens, mask = problem(2, 2, 4, 1, (1, 48, 40), MASK_READOUT_INVARIANT, seed=n_iter)
    check(oracle, d, z, y, sens, mask, mu, n_iter, "rank2 k=%d mu=%g" % (n_iter, mu))


@pytest.mark.parametrize("case", [
    (2, 3, 3, 2, (1, 20, 46), MASK_READOUT_INVARIANT, 1, False),     # per-frame sensitivities, three examples
    (2, 2, 3, 2, (1, 64, 46), MASK_FULL, 0, True),                   # full weighted mask
    (3, 2, 3, 1, (6, 64, 32), MASK_READOUT_INVARIANT, 0, False),     # row-tile 3-D path
    (3, 1, 2, 2, (4, 6, 8), MASK_FULL, 1, False),
    (3, 2, 3, 1, (10, 46, 32), MASK_READOUT_INVARIANT, 0, True),
    (2, 1, 2, 1, (1, 2, 2), MASK_READOUT_INVARIANT, 0, False),       # smallest supported image
    (2, 2, 3, 2, (1, 16, 320), MASK_READOUT_INVARIANT, 0, False),    # three-stage row plan: <p,q> by its own kernel
    (2, 3, 2, 1, (1, 10, 160), MASK_READOUT_INVARIANT, 0, True),     # <p,q> per row from the operator, ragged line groups
])
def test_shapes_and_masks(oracle, case):
    rank, B, C, T, n, kind, shf, weighted = case
    d, z, y, sens, mask = problem(rank, B, C, T, n, kind, sens_has_frames=shf, weighted=weighted, seed=sum(n))
    check(oracle, d, z, y, sens, mask, 0.05, 10, "case %s" % (case,))


def test_in_place_and_determinism(oracle):
    d, z, y, sens, mask = problem(2, 2, 3, 2, (1, 32, 24), MASK_READOUT_INVARIANT, seed=4)
    check(oracle, d, z, y, sens, mask, 0.05, 6, "in place", in_place=True)
    a = run_gpu_modl(z, y, sens, mask, 0.05, 10, 2, 0, MASK_READOUT_INVARIANT)
    b = run_gpu_modl(z, y, sens, mask, 0.05, 10, 2, 0, MASK_READOUT_INVARIANT)
    assert np.array_equal(a.view(np.float32), b.view(np.float32))


def test_examples_are_independent_systems(oracle):
    """An example's result does not depend on the rest of the batch."""
    d, z, y, sens, mask = problem(2, 3, 3, 1, (1, 32, 24), MASK_READOUT_INVARIANT, seed=9)
    z[1] *= 50.0                                         # a very different scale in the middle example
    both = run_gpu_modl(z, y, sens, mask, 0.05, 5, 2, 0, MASK_READOUT_INVARIANT)
    for b in range(3):
        alone = run_gpu_modl(z[b:b + 1], y[b:b + 1], sens[b:b + 1], mask[b:b + 1], 0.05, 5, 2, 0, MASK_READOUT_INVARIANT)
        close(both[b:b + 1], alone.astype(np.complex128), "example %d" % b)


def test_degenerate_inputs():
    d, z, y, sens, mask = problem(2, 2, 2, 1, (1, 8, 8), MASK_READOUT_INVARIANT, seed=1)
    out = run_gpu_modl(np.zeros_like(z), np.zeros_like(y), sens, mask, 0.05, 10, 2, 0, MASK_READOUT_INVARIANT)
    assert np.all(out == 0)                              # zero right-hand side: exactly zero, no NaN
    out = run_gpu_modl(z, y, sens, mask, 0.05, 0, 2, 0, MASK_READOUT_INVARIANT)
    assert np.all(out == 0)                              # no steps: the starting point
    zz = z.copy(); zz[1] = 0; yy = y.copy(); yy[1] = 0   # one example with a zero right-hand side
    out = run_gpu_modl(zz, yy, sens, mask, 0.05, 4, 2, 0, MASK_READOUT_INVARIANT)
    assert np.all(out[1] == 0) and np.isfinite(out.view(np.float32)).all() and np.abs(out[0]).max() > 0


def test_identity_normal_operator():
    """Full mask, unit-norm sensitivities: A^H A = I, so grad_z = mu / (1 + mu) g after one step."""
    d, z, y, sens, mask = problem(2, 2, 4, 1, (1, 64, 46), MASK_READOUT_INVARIANT, seed=3)
    mask[:] = 1.0
    mu = 0.7
    got = run_gpu_modl(z, None, sens, mask, mu, 1, 2, 0, MASK_READOUT_INVARIANT)
    close(got, mu / (1 + mu) * z.astype(np.complex128), "identity")


@pytest.mark.parametrize("name,mu", [("slice64", 0.05), ("knee2d", 0.05), ("knee2d", 4.0), ("cine", 0.05)])
def test_workloads_ten_steps(oracle, name, mu):
    """The paper's MoDL settings: 10 CG steps, mu = 0.05 (R = 16, and the cine network) or 4.0 (R = 4),
    on the knee-like 2-D workload and the cine workload at full size."""
    w, d, inp, mask, y = workload_case(oracle, name)
    ref = oracle.modl_cg_forward(inp["x"], y, inp["sens"], mask, mu, 10, d, nthreads=8)
    got = run_gpu_modl(inp["x"], y, inp["sens"], mask, mu, 10, w.fft_rank, 0, MASK_READOUT_INVARIANT)
    close(got, ref, name + " solve")
    refv = oracle.modl_cg_vjp(inp["g"], inp["sens"], mask, mu, 10, d, nthreads=8)
    gotv = run_gpu_modl(inp["g"], None, inp["sens"], mask, mu, 10, w.fft_rank, 0, MASK_READOUT_INVARIANT)
    close(gotv, refv, name + " vjp")


def test_error_codes():
    import torch
    import paper_2207_08393_b200 as g
    from paper_2207_08393_b200 import binding
    dev = torch.device("cuda:0")
    z = torch.zeros((1, 1, 1, 8, 8), dtype=torch.complex64, device=dev)
    y = torch.zeros((1, 2, 1, 1, 8, 8), dtype=torch.complex64, device=dev)
    s = torch.zeros((1, 2, 1, 8, 8), dtype=torch.complex64, device=dev)
    m = torch.ones((1, 1, 8), dtype=torch.float32, device=dev)
    out = torch.empty_like(z)
    probe = g.make_dims(1, 2, 1, 2, (1, 8, 8))
    nbytes = g.gleam_modl_cg_workspace_size(probe)
    assert nbytes > g.gleam_dc_workspace_size(probe) + 3 * z.numel() * 8
    ws = torch.empty(nbytes, dtype=torch.uint8, device=dev)
    d = g.make_dims(1, 2, 1, 2, (1, 8, 8), stream=torch.cuda.current_stream(), workspace=ws)
    for mu, n_iter in ((0.0, 10), (-1.0, 10), (float("nan"), 10), (0.05, -1), (0.05, 1001)):
        with pytest.raises(g.GleamError) as e:
            g.gleam_modl_cg_forward(z, y, s, m, mu, n_iter, out, d)
        assert e.value.status == binding.GLEAM_ERR_BAD_DIMS
    small = g.make_dims(1, 2, 1, 2, (1, 8, 8), workspace=ws.data_ptr(), workspace_bytes=nbytes - 256)
    with pytest.raises(g.GleamError) as e:
        g.gleam_modl_cg_forward(z, y, s, m, 0.05, 10, out, small)
    assert e.value.status == binding.GLEAM_ERR_WORKSPACE_TOO_SMALL
    with pytest.raises(g.GleamError) as e:
        g.gleam_modl_cg_forward(z, None, s, m, 0.05, 10, out, d)
    assert e.value.status == binding.GLEAM_ERR_NULL_POINTER
    with pytest.raises(g.GleamError) as e:                       # output inside the workspace
        g.gleam_modl_cg_forward(z, y, s, m, 0.05, 10, ws.data_ptr() + 512, d)
    assert e.value.status == binding.GLEAM_ERR_ALIAS
    g.gleam_modl_cg_forward(z, y, s, m, 0.05, 10, z, d)          # exact alias is allowed
    torch.cuda.synchronize()



# sums of the operator: per block and example where one block per SM holds several line groups (two and three examples in a
# block, groups split by coils over four warps, whole ones), per row otherwise (single-warp blocks, four examples, groups with lines
# of two examples); more and fewer sums than a step deals to its warps
@pytest.mark.parametrize("shape,threads,dealt", [
    ((1, 3, 10, 192, 160), 32, False),        # 960 groups of two lines: a sum per row, 1920 of them
    ((2, 5, 8, 160, 160), 384, True),         # 1280 groups, 9 per SM, the last one by four warps
    ((3, 4, 6, 160, 160), 512, True),         # 1440 groups, 10 per SM, two of them by four warps
    ((2, 2, 11, 160, 160), 384, True),        # 1760 groups, 12 per SM
    ((3, 3, 5, 160, 160), 288, True),         # 1200 groups, 9 per SM, too few coils to split
    ((4, 3, 8, 80, 160), 288, True),          # four examples: a sum per row, 640 of them
    ((3, 4, 31, 46, 48), 256, False),         # 1070 groups of four lines, 1426 rows per example
    ((2, 6, 1, 640, 512), 128, True)])       # 1280 groups on 1184 warps: the last ones by four warps each
def test_sums_of_the_operator_and_examples_of_unlike_scale(oracle, shape, threads, dealt):
    import torch
    import paper_2207_08393_b200 as g
    from tests.test_gpu_dispatch import captured
    B, C, T, n1, n2 = shape
    d, z, y, sens, mask = problem(2, B, C, T, (1, n1, n2), MASK_READOUT_INVARIANT, seed=sum(shape), density=0.3)
    scale = np.array([1.0, 300.0, 0.01, 20.0], dtype=np.float32)[:B]
    z *= scale[:, None, None, None, None]
    y *= scale[:, None, None, None, None, None]
    got = run_gpu_modl(z, y, sens, mask, 0.05, 4, 2, 0, MASK_READOUT_INVARIANT)
    gotv = run_gpu_modl(z, None, sens, mask, 0.05, 4, 2, 0, MASK_READOUT_INVARIANT)
    ref = oracle.modl_cg_forward(z, y, sens, mask, 0.05, 4, d, nthreads=8)
    refv = oracle.modl_cg_vjp(z, sens, mask, 0.05, 4, d, nthreads=8)
    for b in range(B):
        close(got[b], ref[b], "%s example %d solve" % (shape, b))
        close(gotv[b], refv[b], "%s example %d vjp" % (shape, b))
    dev = torch.device("cuda:0")
    cg = g.ModlCG(B, C, T, 2, (1, n1, n2))
    tz, ts, tm = (torch.from_numpy(a).to(dev) for a in (z, sens, mask))
    launches = captured(lambda: cg.solve_vjp(tz, ts, tm, 0.05))
    operator = [k for k in launches if "warpflat_kernel" in k["name"]]
    steps = [k for k in launches if "cg_step_kernel" in k["name"]]
    assert len(operator) == len(steps) == 10 and all(k["threads"] == threads for k in operator), operator[0]
    assert all("cg_step_kernelILb1ELb%d" % dealt in k["name"] for k in steps), steps[0]


# vector launches: blocks, and elements that a thread requests at once; two, four and three a thread at once, four in rounds of two; blocks
# that are full, nearly empty and part full at the end, several examples.  Behind an operator of one block per SM (11, 12 and 16
# warps, with and without shared groups, sums per block and per row) four at once unless a block of two fits next to it
@pytest.mark.parametrize("shape,blocks,batch", [
    ((1, 2, 1, 46, 46), 3, 2), ((2, 2, 2, 184, 192), 138, 2), ((1, 2, 3, 320, 160), 75, 4), ((3, 3, 1, 320, 256), 120, 4), ((1, 2, 18, 192, 160), 270, 4),
    ((1, 2, 20, 192, 160), 400, 3), ((1, 2, 22, 192, 160), 440, 3), ((1, 2, 23, 192, 160), 345, 2), ((1, 2, 24, 320, 192), 592, 2),
    ((3, 5, 8, 128, 96), 144, 2),             # 11 warps, sums per block
    ((48, 6, 1, 64, 64), 96, 2),              # 11 warps, sums per row
    ((11, 12, 1, 240, 64), 88, 4),            # 12 warps, a group shared, sums per row
    ((11, 12, 1, 320, 64), 110, 2),           # 12 warps, none shared
    ((1, 4, 10, 256, 80), 100, 2),            # 12 warps, a group shared, sums per block
    ((3, 4, 24, 96, 32), 108, 4),             # 12 warps of 32 points
    ((1, 6, 28, 80, 128), 140, 4),            # 8 warps
    ((1, 10, 7, 512, 80), 140, 4)])           # 16 warps
def test_vector_launches(oracle, shape, blocks, batch):
    import torch
    import paper_2207_08393_b200 as g
    from tests.test_gpu_dispatch import captured
    B, C, T, n1, n2 = shape
    d, z, y, sens, mask = problem(2, B, C, T, (1, n1, n2), MASK_READOUT_INVARIANT, seed=sum(shape), density=0.3)
    close(run_gpu_modl(z, y, sens, mask, 0.5, 3, 2, 0, MASK_READOUT_INVARIANT), oracle.modl_cg_forward(z, y, sens, mask, 0.5, 3, d, nthreads=8), "%s solve" % (shape,))
    cg = g.ModlCG(B, C, T, 2, (1, n1, n2))
    tz, ts, tm = (torch.from_numpy(a).to("cuda:0") for a in (z, sens, mask))
    steps = [k for k in captured(lambda: cg.solve_vjp(tz, ts, tm, 0.5)) if "cg_step_kernel" in k["name"]]
    assert len(steps) == 10 and all(k["blocks"] == blocks and "ELi%dE" % batch in k["name"] for k in steps), steps[0]


def textbook_steps(z, sens, mask, mu, n_iter, dtype):
    """Textbook conjugate gradients on the VJP's system in numpy, vectors in ``dtype``, scalars in double; one coil
    expansion, transforms along the last axis only (a readout-invariant mask).  All iterates."""
    real = np.float32 if dtype == np.complex64 else np.float64
    s, m = sens[0].astype(dtype), np.fft.ifftshift(mask[0].astype(real), axes=-1)[:, None, :]
    inner = lambda a, b: float(np.sum(a.real.astype(np.float64) * b.real + a.imag.astype(np.float64) * b.imag))
    r = (real(mu) * z[0].astype(dtype)).astype(dtype)
    x, p, rr, out = np.zeros_like(r), r.copy(), inner(r, r), []
    for _ in range(n_iter):
        k = np.fft.fft(s[:, None] * p[None], norm="ortho") * (m * m)[None]
        q = (p + real(1 / mu) * np.sum(s.conj()[:, None] * np.fft.ifft(k.astype(dtype), norm="ortho").astype(dtype), axis=0)).astype(dtype)
        alpha = rr / (mu * inner(p, q))
        x = (x + real(alpha) * p).astype(dtype)
        r = (r - real(alpha * mu) * q).astype(dtype)
        rr, last = inner(r, r), rr
        p = (r + real(rr / last) * p).astype(dtype)
        out.append(x)
    return out


@pytest.mark.parametrize("kind", [MASK_READOUT_INVARIANT, MASK_FULL])      # sums from the operator's rows / from their own kernel
def test_step_lengths_of_an_ill_conditioned_system(kind):
    """mu = 1e-4, condition number about 1e4: an error of beta is amplified by it, so the iterates show whether beta is
    as good as one from a residual norm that is summed first.  Bound: twice the error, against 64 bits, of textbook steps
    with vectors in single precision (the rounding of the vectors differs between the two; 7 to 10 times without the
    conjugacy term)."""
    rng = np.random.default_rng(1)
    C, T, n1, n2, mu = 8, 4, 96, 160, float(np.float32(1e-4))
    u1, u2, a = np.linspace(-1, 1, n1)[:, None], np.linspace(-1, 1, n2)[None, :], 2 * np.pi * np.arange(C)[:, None, None] / C
    sens = np.exp(-(u1 - np.cos(a)) ** 2 - (u2 - np.sin(a)) ** 2) * np.exp(1j * (a + u1))
    sens = (sens / np.sqrt(np.sum(np.abs(sens) ** 2, axis=0)))[None, :, None].astype(np.complex64)      # (B, C, n0, n1, n2)
    mask = (rng.uniform(size=(1, T, n2)) < 0.1).astype(np.float32)
    z = crandn(rng, 1, T, 1, n1, n2)
    single = textbook_steps(z[:, :, 0], sens[:, :, 0], mask, mu, 20, np.complex64)
    double = textbook_steps(z[:, :, 0], sens[:, :, 0], mask, mu, 20, np.complex128)
    given = mask if kind == MASK_READOUT_INVARIANT else np.ascontiguousarray(np.broadcast_to(mask[:, :, None, None, :], (1, T, 1, n1, n2)))
    for k in (10, 15, 20):
        ref = double[k - 1]
        err = lambda v: np.linalg.norm(v.astype(np.complex128) - ref) / np.linalg.norm(ref)
        got = run_gpu_modl(z, None, sens, given, mu, k, 2, 0, kind)
        assert err(got[0, :, 0]) <= 2 * err(single[k - 1]), (k, err(got[0, :, 0]), err(single[k - 1]))

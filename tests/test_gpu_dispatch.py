"""Which kernels and launch shapes the rules of the dispatch choose, read from the captured launches of a call, and the
results of the calls whose choice lies next to a line, against the CPU oracle."""
import ctypes

import pytest

from oracle.oracle import MASK_READOUT_INVARIANT
from tests.gpu_common import assert_close
from tests.test_gpu_parity import problem
from tests.test_gpu_tiles import check_all

pytestmark = pytest.mark.gpu


def captured(fn):
    """The kernel launches of fn(), in order: name, blocks, threads, resident blocks on this GPU, bytes of local memory (spilled
    registers), and whether the launch may start before the one before it has ended."""
    import torch
    from cuda.bindings import driver
    def ok(r):
        assert int(r[0]) == 0, r[0]
        return r[1:] if len(r) > 2 else r[1] if len(r) == 2 else None
    fn()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        fn()
    raw = driver.CUgraph(graph.raw_cuda_graph())
    count = ok(driver.cuGraphGetNodes(raw))[1]
    nodes = ok(driver.cuGraphGetNodes(raw, count))[0]
    # through ctypes: the package gives its buffer of edge data back before they are read
    class Edge(ctypes.Structure):
        _fields_ = [("from_port", ctypes.c_ubyte), ("to_port", ctypes.c_ubyte), ("type", ctypes.c_ubyte), ("reserved", ctypes.c_ubyte * 5)]
    get_edges, edges = ctypes.CDLL("libcuda.so.1").cuGraphGetEdges_v2, ctypes.c_size_t(0)
    get_edges.argtypes = [ctypes.c_void_p] * 4 + [ctypes.POINTER(ctypes.c_size_t)]
    assert get_edges(graph.raw_cuda_graph(), None, None, None, edges) == 0
    before, after, data = (ctypes.c_void_p * edges.value)(), (ctypes.c_void_p * edges.value)(), (Edge * edges.value)()
    assert edges.value == 0 or get_edges(graph.raw_cuda_graph(), before, after, data, edges) == 0
    programmatic = int(driver.CUgraphDependencyType.CU_GRAPH_DEPENDENCY_TYPE_PROGRAMMATIC)
    follows = {b: (a, e.type == programmatic) for a, b, e in zip(before, after, data)}
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    launches = {}
    for n in nodes:
        p = ok(driver.cuGraphKernelNodeGetParams(n))
        f = p.func if int(p.func) else ok(driver.cuKernelGetFunction(p.kern))
        per_sm = ok(driver.cuOccupancyMaxActiveBlocksPerMultiprocessor(f, p.blockDimX, p.sharedMemBytes))
        launches[int(n)] = dict(name=ok(driver.cuFuncGetName(f)).decode(), blocks=p.gridDimX * p.gridDimY, threads=p.blockDimX,
                                resident=per_sm * sms, spilled=ok(driver.cuFuncGetAttribute(driver.CUfunction_attribute.CU_FUNC_ATTRIBUTE_LOCAL_SIZE_BYTES, f)),
                                early=follows.get(int(n), (0, False))[1])
    order = [n for n in launches if n not in follows]
    nexts = {a: b for b, (a, _) in follows.items()}
    while order[-1] in nexts:
        order.append(nexts[order[-1]])
    assert len(order) == len(launches)
    return [launches[n] for n in order]


def holder(shape):
    import torch
    import paper_2207_08393_b200 as g
    B, C, T, n1, n2 = shape
    n, dev = (1, n1, n2), torch.device("cuda:0")
    x = torch.zeros((B, T) + n, dtype=torch.complex64, device=dev)
    y = torch.zeros((B, C, T) + n, dtype=torch.complex64, device=dev)
    s = torch.zeros((B, C) + n, dtype=torch.complex64, device=dev)
    m = torch.ones((B, T, n2), dtype=torch.float32, device=dev)
    return g.DataConsistency(B, C, T, 2, n), x, y, s, m


# (batch, coils, frames, n1, n2), rounds that the kernel with the coils side by side may take
@pytest.mark.parametrize("shape,most", [
    ((1, 7, 1, 320, 512), 1), ((1, 7, 1, 320, 320), 1), ((1, 6, 1, 320, 384), 1), ((1, 12, 1, 192, 640), 1),
    ((1, 12, 1, 184, 184), 1), ((1, 12, 1, 192, 92), 1), ((1, 40, 1, 512, 256), 2), ((2, 16, 1, 512, 256), 2),
    ((1, 12, 1, 184, 368), 2), ((1, 14, 1, 320, 240), 2), ((1, 8, 1, 64, 64), 1)])
def test_rounds_of_the_coils_side_by_side(shape, most):
    dc, x, y, s, m = holder(shape)
    for fn in (lambda: dc.vjp(x, s, m, 1.0), lambda: dc.forward(x, y, s, m, 1.0), lambda: dc.adjoint(y, s, m)):
        row = captured(fn)[-1]
        if "coilpar_kernel" in row["name"]:
            assert -(-row["blocks"] // row["resident"]) <= most, row
        else:
            assert shape[3:] != (64, 64), row              # few lines


@pytest.mark.parametrize("shape", [(1, 7, 1, 320, 320), (1, 12, 1, 192, 92), (1, 12, 1, 184, 368), (1, 14, 1, 320, 240),
                                   (1, 12, 1, 384, 160), (1, 40, 1, 160, 256)])
def test_results_next_to_the_lines(oracle, shape):
    B, C, T, n1, n2 = shape
    d, x, y, sens, mask = problem(2, B, C, T, (1, n1, n2), MASK_READOUT_INVARIANT, weighted=(C == 14), seed=n1 + n2, density=0.3)
    check_all(oracle, d, x, y, sens, mask, 0.9, "%s" % (shape,))


# the z table starts early unless a row launch of one round that lets it in at its start may lie before it (single-warp blocks
# with numbered units and z do not): line groups against the resident blocks of 148 SMs, with and without z
@pytest.mark.parametrize("shape,early", [
    ((2, 16, 1, 640, 320), False),           # one round each
    ((3, 15, 1, 640, 368), False),           # 1920 groups with z, 960 without: the VJP call is one round
    ((5, 8, 1, 640, 240), False),            # 1600 groups, 1628 blocks
    ((3, 16, 1, 640, 320), True),            # 1920 groups, 1480 and 1776 blocks
    ((1, 8, 24, 192, 160), True),            # 2304 groups, 2072 blocks
    ((11, 6, 1, 320, 256), True),            # 1760 groups, 1776 blocks with z (numbered units), 1628 without
    ((4, 8, 8, 64, 64), False),              # 512 groups of the plain kernel with z, 1024 of numbered units without
    ((1, 8, 1, 64, 64), True)])              # a few blocks
def test_early_start_of_the_z_table(shape, early):
    dc, x, y, s, m = holder(shape)
    launches = captured(lambda: (dc.forward(x, y, s, m, 1.0), dc.vjp(x, s, m, 1.0), dc.forward(x, y, s, m, 1.0)))
    tables = [i for i, k in enumerate(launches) if "col_z_kernel" in k["name"]]
    assert len(tables) == 2 and len(launches) == 5
    assert launches[tables[1]]["early"] == early, launches[tables[1]]
    assert all(k["early"] for i, k in enumerate(launches) if i > 0 and i not in tables)


# last round of the row kernel: groups shared by the four warps of a block (even and odd numbers of coils, one and two lines a
# group, a last group with a line past the end, behind one and two full rounds), calls that keep single-warp blocks next to the lines
@pytest.mark.parametrize("shape,shared", [
    ((4, 6, 1, 640, 368), ("vjp", "aty", "prepared", "adjoint")),       # 1280 groups of two lines and 2560 of one, 1184 warps
    ((2, 13, 1, 640, 512), ("vjp", "aty", "prepared")),                 # 1280 groups, weighted mask (A^H y: more warps an SM)
    ((7, 6, 1, 368, 512), ("prepared",)),                               # 2576 groups: two full rounds
    ((2, 7, 3, 320, 640), ()),                                          # 1920 groups: three a block
    ((2, 7, 1, 640, 640), ("vjp", "aty", "prepared", "adjoint")),       # 1280 groups
    ((4, 5, 1, 640, 368), ()),                                          # too few coils
    ((27, 12, 3, 46, 256), ("prepared", "adjoint")),                    # 1863 groups of two lines, 1776 warps
    ((23, 13, 5, 46, 96), ("prepared",)),                               # 2645 groups, 2368 warps
    ((27, 10, 3, 46, 256), ())])                                        # too few coils for 12 warps an SM
def test_last_round_of_the_row_kernel(oracle, shape, shared):
    import torch
    B, C, T, n1, n2 = shape
    d, x, y, sens, mask = problem(2, B, C, T, (1, n1, n2), MASK_READOUT_INVARIANT, weighted=(C == 13), seed=sum(shape), density=0.3)
    check_all(oracle, d, x, y, sens, mask, 0.9, "%s" % (shape,))
    dc, tx, ty, ts, tm = holder(shape)
    zero = torch.zeros_like(tx)
    for name, fn in (("vjp", lambda: dc.vjp(tx, ts, tm, 1.0)), ("aty", lambda: dc.forward_aty(tx, zero, ts, tm, 1.0)),
                     ("prepared", lambda: dc.forward_prepared(tx, ty, ts, tm, 1.0)), ("adjoint", lambda: dc.adjoint(ty, ts, tm))):
        row = [k for k in captured(fn) if "warpflat_kernel" in k["name"] or "warpline_kernel" in k["name"]][-1]
        assert (row["threads"] == 128) == (name in shared), (name, row)
    dev = torch.device("cuda:0")
    t = [torch.from_numpy(a).to(dev) for a in (x, y, sens, mask)]
    aty = dc.adjoint(t[1], t[2], t[3])
    got = dc.forward_aty(t[0], aty, t[2], t[3], 0.9).cpu().numpy()
    assert_close(got, oracle.dc_forward(x, y, sens, mask, 0.9, d, nthreads=8), x, "%s normal equations" % (shape,))


# the shared last round with sensitivities that move with the frames, in place (four warps read the rows that one of them writes) and in
# the two-channel layout, bit for bit as the complex calls
@pytest.mark.parametrize("shape", [(4, 7, 2, 320, 368), (1, 6, 4, 320, 640), (4, 9, 2, 160, 512)])
def test_shared_last_round_in_place_and_in_channels(oracle, shape):
    import torch
    import paper_2207_08393_b200 as g
    from tests.test_gpu_bridge import _run
    B, C, T, n1, n2 = shape
    d, x, y, sens, mask = problem(2, B, C, T, (1, n1, n2), MASK_READOUT_INVARIANT, sens_has_frames=1, seed=sum(shape), density=0.3)
    dc = g.DataConsistency(B, C, T, 2, (1, n1, n2), 1)
    t = [torch.from_numpy(a).to("cuda:0") for a in (x, y, sens, mask)]
    dc.prepare(t[1], t[3])
    for fn in (lambda: dc.vjp(t[0], t[2], t[3], 1.0), lambda: dc.forward_prepared(t[0], t[1], t[2], t[3], 1.0)):
        assert captured(fn)[-1]["threads"] == 128
    both, x_ch = g.GLEAM_X_CHANNELS | g.GLEAM_OUT_CHANNELS, oracle.complex_to_channels(x)
    for yy in (y, None):
        plain = _run(d, x, yy, sens, mask, 0.9, 0)
        ref = oracle.dc_forward(x, yy, sens, mask, 0.9, d, nthreads=8) if yy is not None else oracle.dc_vjp(x, sens, mask, 0.9, d, nthreads=8)
        assert_close(plain, ref, x, "moving coils %s" % (shape,))
        assert _run(d, x, yy, sens, mask, 0.9, 0, in_place=True).tobytes() == plain.tobytes()
        plain_ch = oracle.complex_to_channels(plain).tobytes()
        assert _run(d, x_ch, yy, sens, mask, 0.9, both).tobytes() == plain_ch
        assert _run(d, x_ch, yy, sens, mask, 0.9, both, in_place=True).tobytes() == plain_ch


# prepared steps of 512 points share the groups of the last round behind at most six full ones, of 368 and 640 points behind any number
@pytest.mark.parametrize("shape,shared", [((23, 6, 1, 320, 512), True), ((26, 6, 1, 320, 512), False), ((23, 6, 1, 320, 640), True), ((23, 6, 1, 320, 368), True)])
def test_rounds_before_a_shared_one(shape, shared):
    dc, x, y, s, m = holder(shape)
    row = [k for k in captured(lambda: dc.forward_prepared(x, y, s, m, 1.0)) if "warpflat_kernel" in k["name"]][-1]
    assert (row["threads"] == 128) == shared, row


# z table: more sampled tiles than blocks (a block walks over several, also with the last tile part full) and fewer, one-, two-
# and three-stage readouts, staged and direct tiles
@pytest.mark.parametrize("rank,coils,n,density", [
    (3, 4, (4, 256, 160), 0.9), (3, 9, (16, 184, 184), 0.95), (3, 3, (46, 96, 120), 0.97), (3, 2, (64, 46, 24), 0.03), (3, 8, (368, 10, 46), 0.5),
    (2, 40, (1, 640, 96), 1.0), (2, 40, (1, 184, 160), 0.9), (2, 3, (1, 320, 368), 0.9), (2, 24, (1, 16, 512), 0.8)])
def test_z_table_tiles_and_blocks(oracle, rank, coils, n, density):
    d, x, y, sens, mask = problem(rank, 1, coils, 1, n, MASK_READOUT_INVARIANT, weighted=(coils % 2 == 1), seed=sum(n), density=density)
    check_all(oracle, d, x, y, sens, mask, 0.8, "z table %s" % (n,))


@pytest.mark.parametrize("n0", [48, 64, 128, 160, 184, 192, 240, 256])
def test_readout_pass_keeps_its_columns_in_registers(n0):
    import torch
    import paper_2207_08393_b200 as g
    n, dev = (n0, 4, 24), torch.device("cuda:0")
    x = torch.zeros((1, 1) + n, dtype=torch.complex64, device=dev)
    y = torch.zeros((1, 2, 1) + n, dtype=torch.complex64, device=dev)
    s = torch.zeros((1, 2) + n, dtype=torch.complex64, device=dev)
    m = torch.ones((1, 1) + n, dtype=torch.float32, device=dev)
    dc = g.DataConsistency(1, 2, 1, 3, n, 0, g.GLEAM_MASK_FULL)
    for fn in (lambda: dc.forward(x, y, s, m, 1.0), lambda: dc.vjp(x, s, m, 1.0), lambda: dc.adjoint(y, s, m)):
        passes = [k for k in captured(fn) if "axis_kernel" in k["name"]]
        assert len(passes) == 1 and passes[0]["spilled"] == 0, passes


# arbitrary masks of volumes: sizes that the bricks take, and ones that they decline (16 x 15 points, single-stage readout or ky,
# radix 32 of ky, 23 points of ky alone, A^H y of 40 points)
@pytest.mark.parametrize("n,brick,adjoint", [((96, 160, 10), True, True), ((40, 48, 12), True, False), ((240, 24, 6), False, False),
                                             ((20, 48, 6), False, False), ((96, 8, 12), False, False), ((64, 384, 4), False, False), ((48, 92, 6), False, False)])
def test_counted_launches_are_the_launches(n, brick, adjoint):
    import torch
    import paper_2207_08393_b200 as g
    dev = torch.device("cuda:0")
    x = torch.zeros((1, 1) + n, dtype=torch.complex64, device=dev)
    y = torch.zeros((1, 2, 1) + n, dtype=torch.complex64, device=dev)
    s = torch.zeros((1, 2) + n, dtype=torch.complex64, device=dev)
    m = torch.ones((1, 1) + n, dtype=torch.float32, device=dev)
    dc = g.DataConsistency(1, 2, 1, 3, n, 0, g.GLEAM_MASK_FULL)
    for fn, taken in ((lambda: dc.forward(x, y, s, m, 1.0), brick), (lambda: dc.vjp(x, s, m, 1.0), brick), (lambda: dc.adjoint(y, s, m), adjoint)):
        launches = captured(fn)
        before = g.gleam_dc_launch_count()
        fn()
        assert g.gleam_dc_launch_count() - before == len(launches), launches
        assert any("brick_kernel" in k["name"] for k in launches) == taken, launches

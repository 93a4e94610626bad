"""GPU parity of the kernels' cuts at the edges of their tiles: CTAs that share a tile of the SINT4 GEMM, the MX GEMM's tile
widths alone and in pairs of CTAs, and the quantizer's row tiles and K chunks."""
import numpy as np
import pytest

from paper_2604_18117_b200 import binding as B
from tests import test_gpu_mxfp as MXFP
from tests import test_gpu_mxint4 as MXINT4
from tests import test_gpu_mxint8 as MXINT8
from tests import test_gpu_parity as SINT4

pytestmark = pytest.mark.gpu


@pytest.fixture
def option():
    used = []

    def set_option(name, value, default=0):
        used.append((name, default))
        B.lq_set_option(name, value)

    yield set_option
    for name, default in used:
        B.lq_set_option(name, default)


def _x(rng, M, K):
    X = rng.standard_normal((M, K)).astype(np.float16)
    X[:, rng.choice(K, max(1, K // 50), replace=False)] *= 20
    return X


@pytest.mark.parametrize("split", [0, 1, 2, 4, 8])
@pytest.mark.parametrize("M,K,N,r,branch", [(1, 1152, 136, 32, "w8a8"), (129, 1088, 72, 0, "none"), (127, 8192, 8, 24, "w16a16"),
                                            (128, 512, 200, 16, "w4a8")])
def test_sint4_tiles_shared_by_a_cluster(option, split, M, K, N, r, branch):
    """One row, one short of and beyond a tile of rows, columns of less than a vector's neighbours, an odd number of groups, fewer
    stages than CTAs, a part that is the branch alone."""
    option("gemm_split", split)
    rng = np.random.default_rng(split + M)
    SINT4._check(SINT4._random_layer(rng, K, N, r, branch), _x(rng, M, K),
                 tol32=SINT4.TOL_F32 * (5 if branch == "w16a16" else 1))


@pytest.mark.parametrize("split", [2, 4, 8])
@pytest.mark.parametrize("M", [1, 9, 25, 128])
def test_launches_close_behind_a_shared_tile_find_its_sums_as_they_were(option, split, M):
    """The CTAs of a cluster leave while kernels behind them begin to fill the shared memory that the partial sums were sent from.  Four layers
    in turn, twenty times, have the bits of each by itself; of the parts of a tile some have no row, or all have."""
    import torch
    from tests.helpers import import_oracle_layer

    option("gemm_split", split)
    rng = np.random.default_rng(split + M)
    st, linears = torch.cuda.current_stream().cuda_stream, []
    for K, N, r, branch in ((1152, 1160, 32, "w8a8"), (576, 2048, 0, "none"), (2048, 136, 24, "w16a16"), (1088, 1024, 16, "w4a8")):
        h, _ = import_oracle_layer(SINT4._random_layer(rng, K, N, r, branch))
        B.lq_layer_to_device(h, 0)
        linears.append((h, B.lq_act_create(h, M, 0), torch.from_numpy(_x(rng, M, K)).cuda(), N))

    def forward(h, act, x, N):
        y = torch.full((M, N), float("nan"), device="cuda")
        B.lq_quantize_act(h, x.data_ptr(), M, act, st)
        B.lq_linear_forward(h, act, y.data_ptr(), B.OUT_F32, st)
        return y

    alone = []
    for l in linears:
        alone.append(forward(*l))
        torch.cuda.synchronize()
    chain = [forward(*l) for _ in range(20) for l in linears]
    torch.cuda.synchronize()
    assert B.lq_get_device_status(0)[0] == 0
    assert all(torch.equal(y, alone[i % len(linears)]) for i, y in enumerate(chain))
    for h, act, _, _ in linears:
        B.lq_act_free(act)
        B.lq_layer_free(h)


@pytest.mark.parametrize("pair", [0, 1])
@pytest.mark.parametrize("width", [64, 128, 160, 192, 224])
@pytest.mark.parametrize("main,branch,r", [("mxint4", "none", 0), ("mxint4", "w8a8", 32), ("mxint4", "w16a16", 24), ("mxfp4", "mxfp8", 64),
                                           ("mxint8", "mxint8", 64), ("mxint8", "mxint4", 128)])
def test_mx_tile_widths_alone_and_in_pairs(option, main, branch, r, width, pair):
    """Three row blocks (a pair's second one is missing), the last of them one row; a last tile of eight columns; K beyond the ring."""
    if (width == 160) != (branch == "w8a8") and width >= 160:
        pytest.skip("layers with an integer branch have the widths up to 160, the others all but 160")
    option("gemm_width", width)
    option("gemm_pair", pair, default=1)
    rng = np.random.default_rng(width + pair)
    M, K, N = 257, 1184, 2 * width + 8
    mod = {"mxint4": MXINT4, "mxfp4": MXFP, "mxint8": MXINT8}[main]
    layer = mod._mx_layer(rng, K, N, r, branch) if main == "mxint4" else mod._layer(rng, K, N, r, branch)
    mod._check(layer, _x(rng, M, K))


@pytest.mark.parametrize("groups,stages", [(1, 1), (8, 1), (3, 4), (5, 3), (0, 0), (8, 2), (4, 4)])
@pytest.mark.parametrize("M,K", [(1, 32), (63, 1160), (200, 8192)])
def test_quantizer_cuts(option, groups, stages, M, K):
    """Row tiles of 8 to 64 rows and chunks of one to four stages, on one row, one short of a tile and several tiles; less than a
    stage, a ragged last stage, and the longest K (an integer branch streams the tile twice).  What a launch cannot have - a chunk
    longer than K, more warps than there are - becomes the largest that it can."""
    option("quant_warps", groups)
    option("quant_ctas", stages)
    rng = np.random.default_rng(M)
    X = _x(rng, M, K)
    SINT4._check(SINT4._random_layer(rng, K, 40, 32, "w8a8"), X)
    MXFP._check(MXFP._layer(rng, K, 40, 33, "mxfp8"), X)
    MXINT8._check(MXINT8._layer(rng, K, 40, 40, "mxint8"), X)


def test_static_calls_of_different_layers_share_the_scratch():
    """What an earlier call of another layer left in the padding of the shared record is not read."""
    from oracle import lq_oracle as O
    from tests.helpers import import_oracle_layer, rel_fro
    import torch

    rng = np.random.default_rng(5)
    for M, K, N, r, branch in ((256, 2048, 264, 64, "w16a16"), (130, 72, 40, 8, "w8a8"), (3, 328, 136, 24, "w16a16"), (3, 328, 8, 0, "none")):
        layer, X = SINT4._random_layer(rng, K, N, r, branch), _x(rng, M, K)
        h, _ = import_oracle_layer(layer)
        B.lq_layer_to_device(h, 0)
        x, y = torch.from_numpy(X).cuda(), torch.empty(M, N, device="cuda")
        B.lq_linear_forward_static(h, x.data_ptr(), M, y.data_ptr(), B.OUT_F32, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        B.lq_layer_free(h)
        assert rel_fro(y.cpu().numpy(), O.forward(X, layer)["Y"]) <= SINT4.TOL_F32 * (10 if branch == "w16a16" else 1)


@pytest.mark.parametrize("main,branch,r", [("mxint4", "w8a8", 32), ("mxfp4", "mxfp8", 64)])
def test_pairs_of_ctas_give_the_bits_of_single_ones_every_time(option, main, branch, r):
    """Long K and several tiles per pair, so that stages keep changing hands between the two CTAs: the output is that of single
    CTAs, call after call."""
    import torch
    from tests.helpers import import_oracle_layer, import_oracle_mxfp_layer

    rng = np.random.default_rng(11)
    M, K, N = 2100, 4096, 1160
    layer = MXINT4._mx_layer(rng, K, N, r, branch) if main == "mxint4" else MXFP._layer(rng, K, N, r, branch)
    h, _ = (import_oracle_layer if main == "mxint4" else import_oracle_mxfp_layer)(layer)
    B.lq_layer_to_device(h, 0)
    act = B.lq_act_create(h, M, 0)
    x, st = torch.from_numpy(_x(rng, M, K)).cuda(), torch.cuda.current_stream().cuda_stream
    B.lq_quantize_act(h, x.data_ptr(), M, act, st)

    def forward():
        y = torch.full((M, N), float("nan"), device="cuda")
        B.lq_linear_forward(h, act, y.data_ptr(), B.OUT_F32, st)
        return y

    option("gemm_pair", 0, default=1)
    alone = forward()
    option("gemm_pair", 1, default=1)
    pairs = [forward() for _ in range(20)]
    torch.cuda.synchronize()
    assert B.lq_get_device_status(0)[0] == 0
    assert all(torch.equal(alone, y) for y in pairs)
    B.lq_act_free(act)
    B.lq_layer_free(h)


def _begins_between_sectors(rng, main, branch, r, M, K, N):
    """Rows of Y that begin on 16-byte boundaries only, by their length or by Y's own place, hold the bits of those that begin on
    32-byte ones, and nothing beside them is written."""
    import torch
    from tests.helpers import import_oracle_layer, import_oracle_mxfp_layer

    layer = {"sint4": SINT4._random_layer, "mxint4": MXINT4._mx_layer, "mxfp4": MXFP._layer}[main](rng, K, N, r, branch)
    h, _ = (import_oracle_mxfp_layer if main == "mxfp4" else import_oracle_layer)(layer)
    B.lq_layer_to_device(h, 0)
    act = B.lq_act_create(h, M, 0)
    x, st = torch.from_numpy(_x(rng, M, K)).cuda(), torch.cuda.current_stream().cuda_stream
    B.lq_quantize_act(h, x.data_ptr(), M, act, st)
    for dtype, out in ((torch.float16, B.OUT_F16), (torch.float32, B.OUT_F32)):
        size, got = 16 // torch.empty(0, dtype=dtype).element_size(), []      # elements of 16 bytes
        for at in (2 * size, 3 * size):
            y = torch.full((M * N + 6 * size,), 7.0, dtype=dtype, device="cuda")
            assert y.data_ptr() % 32 == 0
            B.lq_linear_forward(h, act, y.data_ptr() + 16 * at // size, out, st)
            got.append(y[at:at + M * N])
            assert bool((y[:at] == 7).all()) and bool((y[at + M * N:] == 7).all())
        assert torch.equal(got[0], got[1])
        assert float(got[0].float().std()) > 0
    assert B.lq_get_device_status(0)[0] == 0
    B.lq_act_free(act)
    B.lq_layer_free(h)


@pytest.mark.parametrize("main,branch,r", [("sint4", "w8a8", 32), ("mxint4", "w8a8", 32), ("mxfp4", "mxfp8", 64)])
@pytest.mark.parametrize("N", [8, 72, 208])
def test_outputs_that_begin_between_sectors(option, main, branch, r, N):
    option("gemm_split", 1)                                       # (tiles shared by a cluster have stores of their own)
    _begins_between_sectors(np.random.default_rng(N), main, branch, r, 131, 200, N)


@pytest.mark.parametrize("split", [2, 4, 8])
@pytest.mark.parametrize("M", [1, 9, 131])
@pytest.mark.parametrize("N", [8, 72, 208])
def test_outputs_of_shared_tiles_that_begin_between_sectors(option, split, M, N):
    """(parts of a tile without rows, with some and with all)"""
    option("gemm_split", split)
    _begins_between_sectors(np.random.default_rng(N + M), "sint4", "w8a8", 32, M, 1152, N)


@pytest.mark.parametrize("M,K,N", [(2047, 40, 24), (2048, 40, 24), (2049, 40, 24), (2305, 3200, 24), (2300, 40, 3800), (2300, 1152, 1160)])
def test_row_chunks_of_a_call_from_host_memory(M, K, N):
    """Around the number of rows from which chunks differ in size, few bytes and many, row counts beside a tile: the bits of the call on device
    memory, and nothing beside them."""
    import torch
    from tests.helpers import import_oracle_layer

    rng = np.random.default_rng(M)
    h, _ = import_oracle_layer(MXINT4._mx_layer(rng, K, N, 16, "w8a8"))
    B.lq_layer_to_device(h, 0)
    act, st = B.lq_act_create(h, M, 0), torch.cuda.current_stream().cuda_stream
    x = torch.from_numpy(_x(rng, M, K)).pin_memory()
    y, ref = torch.full((M + 1, N), float("nan")).pin_memory(), torch.empty(M, N, device="cuda")
    B.lq_linear_forward_host(h, act, x.data_ptr(), M, y.data_ptr(), B.OUT_F32, st)
    xd = x.cuda()
    B.lq_quantize_act(h, xd.data_ptr(), M, act, st)
    B.lq_linear_forward(h, act, ref.data_ptr(), B.OUT_F32, st)
    assert torch.equal(y[:M], ref.cpu()) and bool(y[M].isnan().all())
    assert B.lq_get_device_status(0)[0] == 0
    B.lq_act_free(act)
    B.lq_layer_free(h)


@pytest.mark.parametrize("ctas", [6, 0])
@pytest.mark.parametrize("width", [64, 0, 192])
@pytest.mark.parametrize("main,branch,r,K", [("mxint4", "none", 0, 1152), ("mxint4", "w8a8", 32, 1152), ("mxint4", "w16a16", 24, 1030 + 2), ("mxfp4", "mxfp8", 64, 1400),
                                             ("mxfp4", "mxfp8", 64, 1152), ("mxint8", "mxint8", 64, 1152), ("mxint8", "mxint4", 128, 1160),
                                             ("mxint8", "mxint4", 128, 1152)])
def test_weights_that_stay_while_a_pair_goes_down_its_columns(option, main, branch, r, K, width, ctas):
    """Runs of tiles that begin and end within a column, change columns once or more often, a pair without a second row block, a last tile of eight
    columns, K at and beyond what stays: the bits of single CTAs."""
    import torch
    from tests.helpers import import_oracle_layer, import_oracle_mxfp_layer, import_oracle_mxint_layer

    rng = np.random.default_rng(K + width)
    M, N = 2600, 1160
    mod = {"mxint4": MXINT4, "mxfp4": MXFP, "mxint8": MXINT8}[main]
    layer = mod._mx_layer(rng, K, N, r, branch) if main == "mxint4" else mod._layer(rng, K, N, r, branch)
    h, _ = {"mxint4": import_oracle_layer, "mxfp4": import_oracle_mxfp_layer, "mxint8": import_oracle_mxint_layer}[main](layer)
    B.lq_layer_to_device(h, 0)
    act = B.lq_act_create(h, M, 0)
    x, st = torch.from_numpy(_x(rng, M, K)).cuda(), torch.cuda.current_stream().cuda_stream
    B.lq_quantize_act(h, x.data_ptr(), M, act, st)
    option("gemm_width", 160 if width == 192 and branch == "w8a8" else width)

    def forward(pair, n):
        option("gemm_pair", pair, default=1)
        option("gemm_ctas", n)
        y = torch.full((M, N), float("nan"), device="cuda")
        B.lq_linear_forward(h, act, y.data_ptr(), B.OUT_F32, st)
        return y

    alone, pairs = forward(0, 0), forward(1, ctas)
    torch.cuda.synchronize()
    assert B.lq_get_device_status(0)[0] == 0
    assert torch.equal(alone, pairs)
    B.lq_act_free(act)
    B.lq_layer_free(h)


@pytest.mark.parametrize("groups", [1, 2, 4, 5])
@pytest.mark.parametrize("M,r", [(7, 8), (33, 24), (70, 64)])
def test_row_tiles_on_either_side_of_32_rows(option, groups, M, r):
    """The down-projection of tiles of up to 32 rows is 64 rows high and lies elsewhere in tensor memory: fp16 and integer factors, ranks of one and more
    blocks, rows of one warp and of two."""
    option("quant_warps", groups)
    rng = np.random.default_rng(M + groups)
    X = _x(rng, M, 1160)
    SINT4._check(SINT4._random_layer(rng, 1160, 40, r, "w16a16"), X, tol32=SINT4.TOL_F32 * 5)
    MXINT4._check(MXINT4._mx_layer(rng, 1160, 40, r, "w6a6"), X)

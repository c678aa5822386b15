"""The allocation-free bias-gradient entry point (alexnet_bias_grad_noalloc).

Some users of the library cannot call cudaMalloc when they need a bias
gradient: a loop in the middle of overlapped steps (an allocation synchronises
the device and would serialise the loader stream with the compute stream), or a
process that has handed all free HBM to the arena.  For them the entry point
keeps its scratch in a fixed 1 MiB array inside the library image.

Checked here: its output against the existing path's (the bias gradient the
step's own backward-weight operation produces) on two calls in a row, and
against a column sum computed on the host in fp64, over sizes that use one
split, several splits with a ragged or an empty last one, and the most splits
and the largest part of the scratch there are; calls of different shapes follow
one another, so that contents a previous call left in the scratch would show."""
import numpy as np
import pytest
import torch

from paper_1412_2302_b200 import synth

pytestmark = pytest.mark.gpu


def host_colsum(rows_bf16):
    return rows_bf16.to(torch.float32).cpu().numpy().astype(np.float64).sum(axis=0)


def test_bias_grad_noalloc_matches_step_operation_twice():
    from paper_1412_2302_b200 import alexnet as A
    B, seed = 3, synth.BASE_SEED + 7
    net = A.AlexNet(batch=B, seed=seed)
    off = {"conv5.b": (2333824, 256), "conv4.b": (1891072, 384)}
    for call, (op, tdy, tin, key, C) in enumerate([("CONV5_BWD_WEIGHT", "DA5", "A4", "conv5.b", 256),
                                                   ("CONV4_BWD_WEIGHT", "DA4", "A3", "conv4.b", 384)]):
        dy = synth.bf16_grid(seed, 100 + call, (B, C, 13, 13), -1, 1)
        net.set_tensor(tdy, dy)
        net.set_tensor(tin, synth.bf16_grid(seed, 200 + call, (B, 384, 13, 13), -1, 1))
        net.run_op(op)
        net.sync()
        o, n = off[key]
        want = net.get_params(0, 2)[o:o + n]                     # the existing path
        rows = torch.from_numpy(dy.transpose(0, 2, 3, 1).reshape(-1, C).copy()).to(torch.bfloat16).cuda()
        db = torch.full((C,), float("nan"), device="cuda")
        A.bias_grad_noalloc(rows, db)
        torch.cuda.synchronize()
        got = db.cpu().numpy()
        assert np.isfinite(got).all()
        assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want), call
        assert np.linalg.norm(got - host_colsum(rows)) <= 1e-5 * np.linalg.norm(want), call
    # sizes beyond the fixed scratch are refused with a message, nothing is launched
    big = torch.zeros(4, 8192, dtype=torch.bfloat16, device="cuda")
    with pytest.raises(A.AlexNetError) as e:
        A.bias_grad_noalloc(big, torch.zeros(8192, device="cuda"))
    assert e.value.code == A.ERR_ARG and "4096" in str(e.value)
    net.close()


# (rows, channels): splits = clamp(rows / 64, 1, 592 / ceil(channels / 64)), the scratch is laid out [split][channels]
CASES = [(20000, 4096),     # 9 splits (capped from 312) at the largest channel count
         (300, 4096),       # 4 splits right after: only the first four rows of the scratch may be read
         (5000, 4096),      # 9 splits of 556 rows, the last with 552
         (1000, 8),         # 15 splits of 67 rows, the last with 62; the smallest channel count
         (21632, 256),      # 148 splits (capped from 338): conv5's gradient at batch 128
         (777, 72),         # 12 splits; channels not a multiple of 64 (the second column block is partial), rows % 32 != 0
         (1, 4096),         # a single row
         (40000, 64),       # 592 splits of 68 rows, the last ones empty, in one column group: the most scratch there is
         (6500, 64),        # 101 splits of 65 rows, the last one empty
         (64, 64), (127, 40),   # one split, of the fewest and of the most rows
         (128, 40)]         # two splits


def test_bias_grad_noalloc_against_host_column_sums():
    from paper_1412_2302_b200 import alexnet as A
    rng = np.random.default_rng(23)
    st = torch.cuda.Stream()
    for rows, C in CASES:
        x = torch.from_numpy((rng.integers(-64, 65, size=(rows, C)) / 64.0).astype(np.float32)).to(torch.bfloat16).cuda()
        want = host_colsum(x)
        db = torch.full((C,), float("nan"), device="cuda")
        torch.cuda.synchronize()
        A.bias_grad_noalloc(x, db, stream=st)
        st.synchronize()
        got = db.cpu().numpy().astype(np.float64)
        assert np.isfinite(got).all(), (rows, C)
        # bf16 multiples of 1/64, fp32 accumulation: sums of up to 20000 such values are exact in fp32
        assert np.abs(got - want).max() <= 1e-5 * max(1.0, np.abs(want).max()), (rows, C, np.abs(got - want).max())
    for bad_rows, bad_c, word in ((0, 64, "rows"), (16, 12, "multiple of 8"), (16, 4104, "4096")):
        x = torch.zeros(max(bad_rows, 1), bad_c, dtype=torch.bfloat16, device="cuda")
        msg = __import__("ctypes").create_string_buffer(256)
        rc = A.load_library().alexnet_bias_grad_noalloc(A._ptr(x), bad_rows, bad_c, A._ptr(torch.zeros(bad_c, device="cuda")), None, msg, 256)
        assert rc == A.ERR_ARG and word in msg.value.decode(), (bad_rows, bad_c, msg.value)


def test_bias_grad_noalloc_after_calls_that_overlapped():
    """Calls that overlap on the GPU (two streams, no order between them, different numbers of row splits) may spoil their own
    sums, as the header says, and nothing else: the ordered calls that follow are exact, eager ones as well as the replay of
    one captured before."""
    from paper_1412_2302_b200 import alexnet as A
    gen = torch.Generator().manual_seed(29)
    x, y, z = ((torch.randint(-64, 65, (rows, 64), generator=gen) / 64.0).to(torch.bfloat16).cuda() for rows in (150000, 9000, 6500))
    db = [torch.empty(64, device="cuda") for _ in range(3)]
    st = [torch.cuda.Stream(), torch.cuda.Stream()]
    A.bias_grad_noalloc(z, db[2], stream=st[0])                      # set up before the capture
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=st[0]):
        A.bias_grad_noalloc(z, db[2], stream=st[0])
    for _ in range(20):
        for _ in range(4):
            A.bias_grad_noalloc(x, db[0], stream=st[0])
            A.bias_grad_noalloc(y, db[1], stream=st[1])
        torch.cuda.synchronize()
        db[2].fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(db[2].cpu().numpy().astype(np.float64), host_colsum(z))
        for t, out in ((y, db[1]), (x, db[0]), (y, db[1])):
            out.fill_(float("nan"))
            torch.cuda.synchronize()
            A.bias_grad_noalloc(t, out, stream=st[0])
            torch.cuda.synchronize()
            # multiples of 1/64: the fp32 sums are exact
            assert np.array_equal(out.cpu().numpy().astype(np.float64), host_colsum(t))


# one split, the most splits (592 of one column group, 296 of two), two groups around the line from which blocks of 512 rows take more than
# one split per SM (75776 rows), wide layers of several splits, and remainders of the row lanes
@pytest.mark.parametrize("rows,C", [(1, 8), (65, 4096), (74, 4096), (781, 384), (782, 384), (4687, 64), (4688, 64), (9473, 64), (20011, 72),
                                    (75776, 104), (76288, 104), (152001, 128), (303200, 8), (1201, 2432), (1201, 3200), (1201, 4096)])
def test_bias_grad_noalloc_block_sizes(rows, C):
    from paper_1412_2302_b200 import alexnet as A
    rng = np.random.default_rng(rows + C)
    x = torch.from_numpy((rng.integers(-64, 65, size=(rows, C)) / 64.0).astype(np.float32)).to(torch.bfloat16).cuda()
    db = torch.full((C,), float("nan"), device="cuda")
    for _ in range(2):
        A.bias_grad_noalloc(x, db)
        torch.cuda.synchronize()
        # multiples of 1/64 below 2^18 in all: 32-bit sums are exact in any order
        assert np.array_equal(db.cpu().numpy().astype(np.float64), host_colsum(x)), (rows, C)

"""The evaluation pass through the C ABI (alexnet_eval_batch) against the fp64 oracle: centre crop without flip,
dropout replaced by its expectation, logits within rel-L2 2e-2, and the top-1 / top-5 counts exact for the logits the
GPU produced (integer work) and equal to the oracle's wherever the oracle's ranking is not a near-tie."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1412_2302_b200 import synth

pytestmark = pytest.mark.gpu
TOL = 2e-2


def rel(a, b):
    a, b = np.asarray(a, np.float64).ravel(), np.asarray(b, np.float64).ravel()
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


@pytest.mark.parametrize("inverted", [False, True])
def test_eval_batch_against_oracle(inverted):
    from paper_1412_2302_b200 import alexnet as A
    seed, B = synth.BASE_SEED + 31, 12
    mean = synth.mean_image(seed)
    net = A.AlexNet(batch=B, seed=seed, mean_image=mean, flags=A.FLAG_INVERTED_DROPOUT if inverted else 0)
    w = synth.init_params(seed, variance_preserving=True, bias=0.1)
    net.set_params(w)
    img = synth.images(seed, 0, 0, B)
    onet = O.OracleNet(O.OracleConfig(seed=seed, inverted_dropout=inverted), w.astype(np.float64))
    E = O.evaluate(onet, img, np.zeros(B, np.int32), mean)
    # labels at chosen oracle ranks: 0 (top-1), 2 and 4 (top-5 only), 5 and 40 (neither)
    order = np.argsort(-E["z"], axis=1, kind="stable")
    ranks = np.array([0, 2, 4, 5, 40, 0, 1, 4, 5, 7, 0, 3])
    lab = order[np.arange(B), ranks].astype(np.int32)
    E = O.evaluate(onet, img, lab, mean)
    assert E["top1"].sum() == 3 and E["top5"].sum() == 8
    t1, t5, loss = net.eval_batch(0, torch.from_numpy(img).pin_memory(), torch.from_numpy(lab).pin_memory())
    assert np.array_equal(net.get_tensor("CROPFLIP").reshape(B, 3), np.tile([14, 14, 0], (B, 1)))
    for k in ("x0", "f6", "f7", "z"):
        assert rel(net.get_tensor(k.upper()), E[k]) < TOL, k
    assert abs(loss - E["loss"]) < 2e-2 * max(1.0, abs(E["loss"]))
    zg = net.get_tensor("Z").reshape(B, 1000)
    # integer work: exact for the GPU's own logits
    assert t1 == int(O.topk_correct(zg, lab, 1).sum()) and t5 == int(O.topk_correct(zg, lab, 5).sum())
    # and the oracle's verdict wherever its ranking is not a near-tie at the cut
    noise = 2.0 * np.abs(zg - E["z"]).max()
    zs = -np.sort(-E["z"], axis=1)
    zl = E["z"][np.arange(B), lab]
    for k, got in ((1, O.topk_correct(zg, lab, 1)), (5, O.topk_correct(zg, lab, 5))):
        want = O.topk_correct(E["z"], lab, k)
        clear = np.minimum(np.abs(zl - zs[:, k - 1]), np.abs(zl - zs[:, k])) > noise     # label far from the k-th / (k+1)-th logit
        clear |= (np.abs(zs[:, k - 1] - zs[:, k]) > noise) & (zl != zs[:, k - 1]) & (zl != zs[:, k])
        assert np.array_equal(got[clear], want[clear]), k
    assert np.array_equal(net.get_params(0, 0), w)           # evaluation leaves the parameters alone
    # a loaded training batch must be consumed first
    net.load_batch_async(0, torch.from_numpy(img).pin_memory(), torch.from_numpy(lab).pin_memory(), 0)
    with pytest.raises(A.AlexNetError) as e:
        net.eval_batch(0, torch.from_numpy(img).pin_memory(), torch.from_numpy(lab).pin_memory())
    assert e.value.code == A.ERR_STATE
    net.train_step(0)
    t1b, t5b, _ = net.eval_batch(0, torch.from_numpy(img).pin_memory(), torch.from_numpy(lab).pin_memory())
    assert 0 <= t1b <= t5b <= B
    net.close()


@pytest.mark.parametrize("B", [55, 56, 57, 129, 193])
def test_eval_in_chunks_agrees_with_one_pass(B):
    """Images in host memory are evaluated in chunks (one up to 67 images, then two, more from 192 on; 129 and 193 do not
    divide evenly), images on the device in one pass.  Each is within TOL of the oracle by the test above: the logits agree within
    2 TOL, the mean loss to the same relative bound (the test below asks for the same bits), and the counts are exact for the
    logits of each."""
    from paper_1412_2302_b200 import alexnet as A
    seed = synth.BASE_SEED + 32
    net = A.AlexNet(batch=B, seed=seed, mean_image=synth.mean_image(seed))
    net.set_params(synth.init_params(seed, variance_preserving=True, bias=0.1))
    gen = torch.Generator().manual_seed(B)
    img = torch.randint(0, 256, (B, 256, 256, 3), dtype=torch.uint8, generator=gen)
    lab = torch.randint(0, 1000, (B,), dtype=torch.int32, generator=gen)
    got = {}
    for where, im, lb in (("host", img.pin_memory(), lab.pin_memory()), ("device", img.cuda(), lab.cuda())):
        torch.cuda.synchronize()
        t1, t5, loss = net.eval_batch(0, im, lb)
        z = net.get_tensor("Z").reshape(B, 1000)
        assert t1 == int(O.topk_correct(z, lab.numpy(), 1).sum()) and t5 == int(O.topk_correct(z, lab.numpy(), 5).sum()), where
        got[where] = z, loss
    assert rel(got["host"][0], got["device"][0]) < 2 * TOL
    assert abs(got["host"][1] - got["device"][1]) < 2 * TOL * max(1.0, abs(got["device"][1]))
    net.close()


@pytest.mark.parametrize("B", [67, 68, 69, 129, 193, 260])
def test_eval_in_chunks_is_bit_for_bit_the_one_pass(B):
    """Around the smallest batch in two chunks, and with chunks that do not divide evenly.  The chunks of an evaluation from host memory take the tiles of the whole batch's launches, so where the images come from does
    not show: logits, counts and loss are those of the one pass over images on the device, bit for bit."""
    from paper_1412_2302_b200 import alexnet as A
    seed = synth.BASE_SEED + 33
    net = A.AlexNet(batch=B, seed=seed, mean_image=synth.mean_image(seed))
    net.set_params(synth.init_params(seed, variance_preserving=True, bias=0.1))
    gen = torch.Generator().manual_seed(B)
    lab = torch.randint(0, 1000, (B,), dtype=torch.int32, generator=gen)
    for _ in range(2):                                 # (a second batch: nothing of the first may show)
        img = torch.randint(0, 256, (B, 256, 256, 3), dtype=torch.uint8, generator=gen)
        got = []
        for im, lb in ((img.pin_memory(), lab.pin_memory()), (img.cuda(), lab.cuda())):
            torch.cuda.synchronize()
            got.append((net.eval_batch(0, im, lb), net.get_tensor("P5"), net.get_tensor("Z")))
        assert got[0][0] == got[1][0]
        assert np.array_equal(got[0][1], got[1][1]) and np.array_equal(got[0][2], got[1][2])
    net.close()


def test_eval_images_where_they_are():
    """Aligned images on the device are read in place, others are copied first, and of pinned images only the crop's rows travel: one
    result.  Before each of them another batch, on the device and misaligned, fills the staging buffer, so that rows which did not travel show."""
    from paper_1412_2302_b200 import alexnet as A
    seed, B = synth.BASE_SEED + 34, 3
    net = A.AlexNet(batch=B, seed=seed, mean_image=synth.mean_image(seed))
    net.set_params(synth.init_params(seed, variance_preserving=True, bias=0.1))
    gen = torch.Generator().manual_seed(B)
    lab = torch.randint(0, 1000, (B,), dtype=torch.int32, generator=gen)
    img = torch.randint(0, 256, (B, 256, 256, 3), dtype=torch.uint8, generator=gen)

    def misaligned(t):
        odd = torch.zeros(t.numel() + 16, dtype=torch.uint8, device="cuda")[5:5 + t.numel()].view(t.shape)
        odd.copy_(t)
        return odd

    got = []
    for im in (img.cuda(), misaligned(img), img.pin_memory(), img):
        other = misaligned(torch.randint(0, 256, img.shape, dtype=torch.uint8, generator=gen))
        torch.cuda.synchronize()
        net.eval_batch(0, other, lab.pin_memory())
        got.append((net.eval_batch(0, im, lab.pin_memory()), net.get_tensor("X0"), net.get_tensor("Z")))
    for g in got[1:]:
        assert g[0] == got[0][0] and np.array_equal(g[1], got[0][1]) and np.array_equal(g[2], got[0][2])
    net.close()


@pytest.mark.parametrize("B", [1, 2, 3, 4, 5])
def test_eval_of_few_images_with_new_labels_every_call(B):
    """Labels at ranks 0, 4 and 5 of the GPU's own logits, other ones every call and in every kind of memory: the counts are those of the labels of
    the call, the loss is the mean cross-entropy of its logits (one image takes a way of its own out of the softmax kernel)."""
    from paper_1412_2302_b200 import alexnet as A
    seed = synth.BASE_SEED + 36
    net = A.AlexNet(batch=B, seed=seed, mean_image=synth.mean_image(seed))
    net.set_params(synth.init_params(seed, variance_preserving=True, bias=0.1))
    img = torch.from_numpy(synth.images(seed, 0, 0, B)).pin_memory()
    net.eval_batch(0, img, torch.zeros(B, dtype=torch.int32).pin_memory())
    z = net.get_tensor("Z").reshape(B, 1000)
    order = np.argsort(-z, axis=1, kind="stable")
    z64 = z.astype(np.float64)
    lse = np.log(np.exp(z64 - z64.max(1, keepdims=True)).sum(1)) + z64.max(1)
    for call, ranks in enumerate(([0], [4], [5], [0, 4], [5, 0], [4, 5], [999, 0], [0])):
        rank = np.array([ranks[i % len(ranks)] for i in range(B)])
        lab = torch.from_numpy(order[np.arange(B), rank].astype(np.int32))
        lab = lab.pin_memory() if call % 3 == 0 else lab.cuda() if call % 3 == 1 else lab
        torch.cuda.synchronize()
        t1, t5, loss = net.eval_batch(0, img, lab)
        assert (t1, t5) == (int((rank < 1).sum()), int((rank < 5).sum())), (ranks, t1, t5)
        want = (lse - z64[np.arange(B), order[np.arange(B), rank]]).mean()
        # 32-bit exponentials and sums of 1000 terms: some 1e-6 of the logits' size
        assert abs(loss - want) < 1e-5 * max(1.0, np.abs(z64).max()), (ranks, loss, want)
        assert np.array_equal(net.get_tensor("Z").reshape(B, 1000), z)
    net.close()


@pytest.mark.parametrize("B", [3, 128, 129, 256, 300, 512, 520])
def test_eval_fc_layers_against_their_inputs(B):
    """fc6 and fc7 of an evaluation against the inputs that the GPU gave them: ReLU, and the expectation of the dropout mask, whether the reduction
    over the k splits runs inside the GEMM (one or several row tiles, 4, 2 or no splits) or, beyond 512 images, as a launch of its own."""
    from paper_1412_2302_b200 import alexnet as A
    seed = synth.BASE_SEED + 37
    net = A.AlexNet(batch=B, seed=seed, mean_image=synth.mean_image(seed))
    w = synth.init_params(seed, variance_preserving=True, bias=0.1)
    off, _ = O.param_offsets()
    rng = np.random.default_rng(B)
    for k in ("fc6.W", "fc7.W"):
        o, n, _ = off[k]
        w[o:o + n] = rng.integers(-16, 17, size=n) / 1024.0      # exact in bf16
    net.set_params(w)
    gen = torch.Generator(device="cuda").manual_seed(B)
    img = torch.randint(0, 256, (B, 256, 256, 3), dtype=torch.uint8, device="cuda", generator=gen)
    lab = torch.zeros(B, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    net.eval_batch(0, img, lab)
    P = O.unpack(w)
    for name, src, dst in (("fc6", "P5", "F6"), ("fc7", "F6", "F7")):
        K, N = O.FC[name]
        W, b = (torch.from_numpy(np.ascontiguousarray(P[name + k])).cuda().double() for k in (".W", ".b"))
        x = torch.from_numpy(net.get_tensor(src)).cuda().double().reshape(B, K)
        ref = 0.5 * torch.relu(x @ W.reshape(N, K).T + b)
        # one rounding to bf16: at most 2^-9 of each value, and 32-bit sums of 9216 terms far below that
        assert rel(net.get_tensor(dst), ref.cpu().numpy()) < 2.0 ** -9 + 1e-5, name
    net.close()


@pytest.mark.parametrize("where", ["pinned", "device", "pageable"])
def test_preprocessing_after_an_evaluation(where):
    """run_op("PREPROCESS") takes the images of the batch loaded last; an evaluation in between, which keeps the rows of its crop at
    most, leaves them alone wherever its own images are."""
    from paper_1412_2302_b200 import alexnet as A
    seed, B = synth.BASE_SEED + 35, 5
    net = A.AlexNet(batch=B, seed=seed, mean_image=synth.mean_image(seed))
    gen = torch.Generator().manual_seed(B)
    lab = torch.randint(0, 1000, (B,), dtype=torch.int32, generator=gen).pin_memory()
    for step in range(3):                              # (both batch slots)
        net.load_batch_async(0, torch.randint(0, 256, (B, 256, 256, 3), dtype=torch.uint8, generator=gen).pin_memory(), lab, step)
        net.train_step(0)
        net.sync()
        want = net.get_tensor("CROPFLIP"), net.get_tensor("X0")
        img = torch.randint(0, 256, (B, 256, 256, 3), dtype=torch.uint8, generator=gen)
        img = img.pin_memory() if where == "pinned" else img.cuda() if where == "device" else img
        torch.cuda.synchronize()
        net.eval_batch(0, img, lab)
        assert not np.array_equal(net.get_tensor("X0"), want[1])
        net.run_op("PREPROCESS")
        net.sync()
        assert np.array_equal(net.get_tensor("CROPFLIP"), want[0]) and np.array_equal(net.get_tensor("X0"), want[1])
    net.close()

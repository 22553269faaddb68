"""Products split over a cluster and the loss inside the last of them, at the edges of their tiles, against the oracle and, for logits
that are infinite or NaN, against the loss's own launch; a block that gives up a wait."""
import numpy as np
import pytest

from parity_util import compare_step, make_pair, rel_err, sync_from_oracle
from paper_2403_11204_b200 import workloads as wl

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-4, "bf16": 2e-2, "tf32": 2e-3}


def arrays(batch, width, n_classes, precision, seed=3):
    g = np.random.default_rng(seed)
    x = g.random((batch, width), dtype=np.float32)
    if precision == "bf16":
        x = wl.from_bf16_bits(wl.to_bf16_bits(x))
    return x, g.integers(0, n_classes, batch).astype(np.int64)


# K split over four CTAs or not at all (TWO_CASES: over two), one tile and several, rows and columns that cut a piece of four; 65 classes
# take the loss's own launch
CASES = [([200, 136, 47], True, "tf32", 1), ([200, 136, 10], True, "bf16", 129), ([1032, 64], True, "tf32", 300),
         ([1032, 65], True, "bf16", 127), ([136, 62], True, "fp32", 129), ([520, 160, 1], True, "fp32", 65),
         ([784, 130], False, "tf32", 257), ([72, 33], False, "bf16", 128), ([2056, 200], False, "fp32", 63), ([160, 201], False, "fp32", 640),
         ([136, 1032, 96, 40], False, "tf32", 31), ([64, 72, 80, 136, 64], False, "bf16", 513)]


@pytest.mark.parametrize("optimizer", ["sgd", "momentum", "adam"])
@pytest.mark.parametrize("widths,final,precision,batch", CASES)
def test_split_products_and_their_loss_at_tile_edges(widths, final, precision, batch, optimizer):
    n = widths[-1] if final else 13
    gpu, ora = make_pair(widths, n, final, precision, optimizer, 1e-3, batch)
    x, cls = arrays(batch, widths[0], n, precision)
    compare_step(gpu, ora, x, cls, precision, TOL[precision])
    if optimizer == "adam":
        sync_from_oracle(gpu, ora)
    m = max(batch - 5, 1)
    compare_step(gpu, ora, x[:m], cls[:m], precision, TOL[precision])       # a partial batch, optimizer state in play
    gpu.close()


# Products whose tiles of 128 x 64 leave room for two CTAs each and not for four: (layers, final, precision, batch, how many run as clusters of
# two; no other product of the step is split).  Forward with the label loss, weight gradient, dgrad, both of the latter without a bias.
TWO_CASES = [([784, 512], False, "tf32", 900, 1), ([1000, 517], False, "tf32", 517, 1), ([2000, 513], False, "bf16", 600, 1),
             ([2000, 130], False, "tf32", 2047, 2), ([1000, 257], False, "bf16", 4001, 1), ([1032, 577, 1030], False, "tf32", 515, 2),
             ([136, 520, 2056], False, "bf16", 601, 1)]


@pytest.mark.parametrize("optimizer", ["sgd", "adam"])
@pytest.mark.parametrize("widths,final,precision,batch,split", TWO_CASES)
def test_products_split_over_two_blocks(widths, final, precision, batch, split, optimizer):
    gpu, ora = make_pair(widths, 13, final, precision, optimizer, 1e-3, batch)
    x, cls = arrays(batch, widths[0], 13, precision)
    before = gpu.product_launches()["tc_splitk"]
    compare_step(gpu, ora, x, cls, precision, TOL[precision])
    assert gpu.product_launches()["tc_splitk"] - before == split
    gpu.close()


def loss_arms(monkeypatch, widths, n_classes, precision, batch, edit, last_relu=False):
    """Loss and gradients of one step with the cross-entropy in the last product's epilogue and as a launch of its own."""
    import torch
    out, launches = [], []
    for separate in ("0", "1"):
        monkeypatch.setenv("SEG_NO_FUSED_LOSS", separate)
        gpu, _ = make_pair(widths, n_classes, True, precision, "sgd", 0.0, batch, last_relu=last_relu)
        L = len(widths) - 1
        W, b = gpu.params(L - 1)
        edit(W, b)
        gpu.set_params(L - 1, W, b)
        x, cls = arrays(batch, widths[0], min(16, n_classes), precision)
        loss = torch.zeros(1, device="cuda")
        xt, ct = torch.from_numpy(x).cuda(), torch.from_numpy(cls.astype(np.int32)).cuda()
        n = gpu.launch_count()
        gpu.train_step(xt.to(torch.bfloat16) if precision == "bf16" else xt, ct, loss)
        gpu.poll()
        launches.append(gpu.launch_count() - n)
        out.append([loss.cpu().numpy()] + [t.cpu().numpy() for l in range(L) for t in gpu.grads(l)])
        gpu.close()
    assert launches[1] == launches[0] + 1, "the first arm did not take the loss into the product"
    return out


@pytest.mark.parametrize("precision,n_classes", [("tf32", 47), ("bf16", 64)])
def test_classes_of_minus_infinity(precision, n_classes, monkeypatch):
    """Logits of -infinity, in whole slices of a row too: no share of the softmax, and no gradient, as in the loss's own launch."""
    def edit(W, b):
        b[16:] = float("-inf")
    out = loss_arms(monkeypatch, [264, 160, n_classes], n_classes, precision, 70, edit)
    for loss, dW0, db0, dW, db in out:
        assert np.isfinite(loss.item()) and np.all(db[16:] == 0) and np.all(np.isfinite(dW))
    for a, b in zip(*out):
        assert rel_err(a, b) <= TOL[precision]


def test_classes_of_minus_infinity_in_fp32():
    import torch
    gpu, _ = make_pair([264, 160, 33], 33, True, "fp32", "sgd", 0.0, 70)
    W, b = gpu.params(1)
    b[16:] = float("-inf")
    gpu.set_params(1, W, b)
    x, cls = arrays(70, 264, 16, "fp32")
    loss = torch.zeros(1, device="cuda")
    gpu.train_step(torch.from_numpy(x).cuda(), torch.from_numpy(cls.astype(np.int32)).cuda(), loss)
    gpu.poll()
    dW, db = gpu.grads(1)
    assert np.isfinite(loss.item()) and torch.all(db[16:] == 0) and torch.all(torch.isfinite(dW))
    gpu.close()


@pytest.mark.parametrize("precision,n_classes,batch", [("tf32", 47, 200), ("bf16", 61, 129)])
@pytest.mark.parametrize("last_relu", [False, True])
@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_infinite_and_nan_logits_as_in_the_losss_own_launch(precision, n_classes, batch, last_relu, value, monkeypatch):
    """A class whose logit is +infinity or NaN: the same gradients are NaN, infinite or finite, whichever kernel forms the loss."""
    def edit(W, b):
        b[21] = value
    fused, own = loss_arms(monkeypatch, [264, 160, n_classes], n_classes, precision, batch, edit, last_relu)
    for a, b in zip(fused, own):
        ok = np.isfinite(b)
        assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.isfinite(a), ok)
        if ok.any():
            assert np.max(np.abs(a[ok] - b[ok])) <= TOL[precision] * max(np.max(np.abs(b[ok])), 1e-30)


@pytest.mark.parametrize("widths,precision,batch", [([200, 136, 47], "tf32", 131), ([72, 136, 64], "bf16", 300), ([264, 33], "tf32", 64)])
def test_cross_entropy_in_the_product_behind_a_relu(widths, precision, batch):
    gpu, ora = make_pair(widths, widths[-1], True, precision, "momentum", 1e-3, batch, last_relu=True)
    x, cls = arrays(batch, widths[0], widths[-1], precision)
    compare_step(gpu, ora, x, cls, precision, TOL[precision])
    gpu.close()


def test_cross_entropy_at_the_row_limit_of_its_products():
    """Four CTAs per 128 rows: 4736 rows fill 148 SMs and still take the loss into the product, one more row takes its own launch."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = 128 * (sms // 4)
    gpu, ora = make_pair([72, 47], 47, True, "tf32", "sgd", 1e-3, rows + 1)
    x, cls = arrays(rows + 1, 72, 47, "tf32")
    counts = []
    for n in (rows, rows + 1):
        before = gpu.launch_count()
        compare_step(gpu, ora, x[:n], cls[:n], "tf32", TOL["tf32"])
        counts.append(gpu.launch_count() - before)
    assert counts[1] == counts[0] + 1
    gpu.close()


@pytest.mark.parametrize("precision", ["tf32", "fp32"])
def test_recovery_clamps_classes_to_the_right_segments(precision):
    """A left segment of more classes than the right one has: an index beyond the right segment's counts as its last class, whichever
    kernel forms the loss."""
    import torch
    from paper_2403_11204_b200 import binding
    from paper_2403_11204_b200.binding import Segment
    x, cls = arrays(150, 72, 47, precision)
    out = []
    for c in (cls, np.minimum(cls, 9)):
        left = Segment([72, 200, 136], 47, False, precision=precision, optimizer="sgd", lr=0.01, max_batch=150)
        right = Segment([136, 160, 10], 10, True, precision=precision, optimizer="sgd", lr=0.01, max_batch=150, segment_id=1)
        left.gen_labels(1, "normal")
        loss = torch.zeros(1, device="cuda")
        binding.recovery_step(left, right, torch.from_numpy(x).cuda(), torch.from_numpy(c.astype(np.int32)).cuda(), loss)
        left.poll()
        out.append([loss.cpu().numpy()] + [t.cpu().numpy() for l in range(2) for t in left.grads(l)])
        left.close()
        right.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("limit_ns", [1_000, 1_000_000, 50_000_000])
def test_a_block_that_gave_up_stays_for_its_peer_and_no_longer(limit_ns):
    """The end of a split product's block whose wait ran out: a peer that sends only afterwards still finds its shared memory (the
    time-out is recorded once that send has landed), and it does not outstay the peer by more than milliseconds."""
    import time
    import torch
    from paper_2403_11204_b200.binding import SegError
    gpu, ora = make_pair([264, 160, 47], 47, True, "tf32", "sgd", 0.01, 70)
    x, cls = arrays(70, 264, 47, "tf32")
    torch.cuda.synchronize()
    for _ in range(2):                               # the first call loads the kernel
        t0 = time.perf_counter()
        gpu.selftest_bounded_wait(limit_ns)
        with pytest.raises(SegError) as e:
            gpu.poll()
        took = time.perf_counter() - t0
        assert e.value.status == 7
    assert limit_ns * 1e-9 <= took <= limit_ns * 1e-9 + 0.25
    gpu.poll()
    compare_step(gpu, ora, x, cls, "tf32", TOL["tf32"])
    gpu.close()


@pytest.mark.parametrize("batch", [900, 1024])
def test_a_short_bf16_forward_product_does_not_take_clusters_of_two(batch):
    """The last layer of 144-336-992-336 (48 tiles, 16 k-blocks) would take 96 SMs as clusters of two, which three handles beside each
    other pay for; the dgrad of the same shape and the weight gradient of layer 0 are split."""
    import torch
    from paper_2403_11204_b200.binding import Segment
    seg = Segment([144, 336, 992, 336], 47, False, precision="bf16", optimizer="sgd", lr=1e-3, max_batch=batch)
    seg.gen_labels(1, "normal")
    seg.train_step(torch.rand(batch, 144, device="cuda").to(torch.bfloat16), torch.zeros(batch, device="cuda", dtype=torch.int32))
    seg.poll()
    assert seg.product_launches()["tc_splitk"] == 2
    seg.close()

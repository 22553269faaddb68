"""Products split over a cluster and the loss inside the last of them, at the edges of their tiles, against the oracle and, for
logits of -infinity, against the loss's own launch."""
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


# K split over 2 and 4 CTAs or not at all, one tile and several, rows and columns that cut a piece of four; 65 classes take the loss's own launch
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


@pytest.mark.parametrize("precision,n_classes", [("tf32", 47), ("bf16", 64), ("fp32", 33)])
def test_classes_of_minus_infinity(precision, n_classes, monkeypatch):
    """Logits of -infinity, in whole slices of a row too: no share of the softmax, and no gradient, as in the loss's own launch."""
    import torch
    out = []
    for separate in ("0", "1"):
        monkeypatch.setenv("SEG_NO_FUSED_LOSS", separate)
        gpu, _ = make_pair([264, 160, n_classes], n_classes, True, precision, "sgd", 0.0, 70)
        W, b = gpu.params(1)
        b[16:] = float("-inf")
        gpu.set_params(1, W, b)
        x, cls = arrays(70, 264, 16, precision)
        loss = torch.zeros(1, device="cuda")
        xt = torch.from_numpy(x).cuda()
        gpu.train_step(xt.to(torch.bfloat16) if precision == "bf16" else xt, torch.from_numpy(cls.astype(np.int32)).cuda(), loss)
        gpu.poll()
        dW, db = gpu.grads(1)
        assert np.isfinite(loss.item()) and torch.all(db[16:] == 0) and torch.all(torch.isfinite(dW))
        out.append([loss.cpu().numpy(), dW.cpu().numpy(), db.cpu().numpy()])
        gpu.close()
    for a, b in zip(*out):
        assert rel_err(a, b) <= TOL[precision]


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

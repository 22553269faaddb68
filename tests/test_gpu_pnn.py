"""The paper's training procedure end to end (Section 2): train the left partition on the
intermediate labels, store its response, train the right partition on it, join - through
seg_train_epochs / seg_forward_dataset, against oracle/pnn.py, loss by loss."""
import os

import numpy as np
import pytest

from oracle import pnn
from paper_2403_11204_b200 import workloads as wl
from parity_util import make_pair, rel_err, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,epochs,label_dist", [("tiny", [1, 1], "normal"), ("tiny", [2, 1], "uniform_kappa")])
def test_two_partition_training_matches_the_oracle(name, epochs, label_dist):
    import torch
    from paper_2403_11204_b200 import binding
    w = wl.WORKLOADS[name]
    n = 1000                                             # 15 full batches of 64 and one of 40
    pairs = [make_pair(s.widths, w.n_classes, s.is_final, w.precision, w.optimizer, w.lr, w.batch,
                       segment_id=s.segment_id, label_dist=label_dist, kappa=10.0) for s in w.segments]
    gpu = [p[0] for p in pairs]
    ora = [p[1] for p in pairs]
    x = wl.features(w, n)
    cls = wl.class_indices(w, n)
    xt, ct = to_device(x, cls, w.precision)
    losses_g, right_in_g = binding.train_partitioned(gpu, xt, ct, w.batch, epochs)
    for seg in gpu:
        seg.poll()
    losses_o, right_in_o = pnn.train_partitioned(ora, x, cls.astype(np.int64), w.batch, epochs)
    for lg, lo in zip(losses_g, losses_o):
        got = lg.cpu().numpy().astype(np.float64)
        assert got.shape == lo.shape
        assert np.max(np.abs(got - lo) / np.abs(lo)) < 1e-3
    assert rel_err(right_in_g.cpu().numpy(), right_in_o) < 1e-3
    for g, o in zip(gpu, ora):
        for l in range(o.n_layers):
            W, b = g.params(l)
            assert rel_err(W.cpu().numpy(), o.W[l]) < 1e-3 and rel_err(b.cpu().numpy(), o.b[l]) < 1e-3
    pred_g = binding.predict(gpu, xt, w.batch).cpu().numpy()
    pred_o = pnn.predict(ora, x, w.batch)
    assert np.mean(pred_g == pred_o) > 0.99              # argmax may differ only on near-ties
    for seg in gpu:
        seg.close()


@pytest.mark.parametrize("precision,backend,tol", [("fp32", "auto", 1e-4), ("bf16", "tcgen05", 2e-2), ("tf32", "tcgen05", 2e-3)])
def test_recovery_step_matches_the_oracle(precision, backend, tol, monkeypatch, capfd):
    """Section 5 (recovery epochs): the left segment trained through the frozen right segment, on a stream of their own,
    where the second step is captured."""
    import torch
    from paper_2403_11204_b200 import binding
    from parity_util import batch_arrays, captured_steps, expected_captures
    w = wl.WORKLOADS["tiny"]
    batch, stream = 200, torch.cuda.Stream()
    monkeypatch.setenv("SEG_DEBUG", "1")
    gl, ol = make_pair([784, 256, 136], 47, False, precision, "momentum", 0.01, batch, segment_id=0, gemm_backend=backend, stream=stream)
    gr, orr = make_pair([136, 72, 47], 47, True, precision, "momentum", 0.01, batch, segment_id=1, gemm_backend=backend, stream=stream)
    x, cls = batch_arrays(w, batch, 784, precision=precision)
    xt, ct = to_device(x, cls, precision)
    right_before = [t for l in range(2) for t in gr.params(l)]
    for step in range(4):                                   # eager, captured, replayed twice
        loss_t = torch.zeros(1, device="cuda")
        torch.cuda.synchronize()
        binding.recovery_step(gl, gr, xt, ct, loss_t)
        gl.poll()
        loss_o = pnn.recovery_step(ol, orr, x, cls.astype(np.int64))
        assert abs(float(loss_t.item()) - loss_o) <= tol * abs(loss_o)
        if step >= 2:
            continue          # two trajectories in reduced precision drift apart: later steps are held to the loss only
        for l in range(2):
            dW, db = gl.grads(l)
            stream.synchronize()
            assert rel_err(dW.cpu().numpy(), ol.dW[l]) <= tol and rel_err(db.cpu().numpy(), ol.db[l]) <= tol
            W, b = gl.params(l)
            stream.synchronize()
            assert rel_err(W.cpu().numpy(), ol.W[l]) <= tol and rel_err(b.cpu().numpy(), ol.b[l]) <= tol
    assert captured_steps(capfd) == expected_captures(1)
    right_after = [t for l in range(2) for t in gr.params(l)]
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(right_before, right_after))       # frozen: bit-identical
    gl.close(); gr.close()


def test_recovery_step_on_the_default_stream_is_captured_and_replayed(monkeypatch, capfd):
    """On the legacy default stream the step of both handles is recorded on a stream of the left one's: the same bits as on an
    ordinary stream, and both handles go on on the stream they were created for."""
    import torch
    from paper_2403_11204_b200 import binding
    from paper_2403_11204_b200.binding import Segment
    from parity_util import batch_arrays, bits_equal, captured_steps, expected_captures
    w = wl.WORKLOADS["tiny"]
    batch = 96
    x, cls = batch_arrays(w, 2 * batch, 72)
    xt, ct = to_device(x, cls, "tf32")
    monkeypatch.setenv("SEG_DEBUG", "1")
    results = []
    for stream in (None, torch.cuda.Stream()):
        left = Segment([72, 200, 136], 47, False, precision="tf32", optimizer="momentum", lr=0.01, max_batch=batch, stream=stream)
        right = Segment([136, 64, 47], 47, True, precision="tf32", optimizer="momentum", lr=0.01, max_batch=batch, segment_id=1,
                        stream=stream)
        left.gen_labels(wl.LABEL_SEED, "normal")
        losses = torch.zeros(61, device="cuda")
        torch.cuda.synchronize()
        for i in range(60):
            lo = (i % 2) * batch
            binding.recovery_step(left, right, xt[lo:lo + batch], ct[lo:lo + batch], losses[i:i + 1])
        assert captured_steps(capfd) == expected_captures(1)
        y = left.forward(xt[:batch])
        right.train_step(y, ct[:batch], losses[60:])
        left.poll()
        right.poll()
        out = [losses, y] + [t for s in (left, right) for l in range(2) for t in s.params(l)]
        torch.cuda.synchronize()
        results.append([t.cpu().numpy() for t in out])
        left.close()
        right.close()
    for a, b in zip(*results):
        assert bits_equal(a, b)


@pytest.mark.parametrize("precision,backend,tol,hidden", [("fp32", "auto", 1e-4, 200), ("fp32", "auto", 1e-4, 96),
                                                          ("bf16", "tcgen05", 2e-2, 200)])
def test_fully_separate_variant_label_rows_as_input(precision, backend, tol, hidden, monkeypatch, capfd):
    """Section 2, last flowchart: a middle partition trained with the previous cut's labels as input and
    its own cut's labels as target; the input rows are gathered by class on the device (by the staging
    kernel, or, hidden = 96, inside the first launch of a small fp32 segment's two-launch step, which has no graph)."""
    import torch
    from oracle import rng as orng
    from parity_util import captured_steps, compare_step, expected_captures
    monkeypatch.setenv("SEG_DEBUG", "1")
    w = wl.WORKLOADS["tiny"]
    m, batch = 47, 150
    prev_labels = orng.gen_labels(wl.LABEL_SEED, 0, m, 136, orng.DIST_UNIFORM_KAPPA, 10.0)     # cut 0: 47 x 136
    gpu, ora = make_pair([136, hidden, 72], m, False, precision, "momentum", 0.01, batch, segment_id=1,
                         gemm_backend=backend, label_dist="uniform_kappa", stream=torch.cuda.Stream())
    cls = wl.class_indices(w, batch)
    sil_t = torch.from_numpy(prev_labels).cuda()
    ct = torch.from_numpy(cls).cuda()
    for step in range(3):                                   # eager, captured, replayed
        loss_t = torch.zeros(1, device="cuda")
        torch.cuda.synchronize()
        gpu.train_step_label_input(sil_t, ct, loss_t)
        gpu.poll()
        loss_o = ora.train_step(prev_labels[cls], cls.astype(np.int64))
        assert abs(float(loss_t.item()) - loss_o) <= tol * abs(loss_o)
        for l in range(2):
            dW, db = gpu.grads(l)
            gpu.stream.synchronize()
            assert rel_err(dW.cpu().numpy(), ora.dW[l]) <= tol and rel_err(db.cpu().numpy(), ora.db[l]) <= tol
            W, b = gpu.params(l)
            gpu.stream.synchronize()
            assert rel_err(W.cpu().numpy(), ora.W[l]) <= tol
    small = hidden <= 128 and precision == "fp32" and os.environ.get("SEG_NO_SMALL_FUSED") != "1"
    assert captured_steps(capfd) == expected_captures(0 if small else 1)
    # an ordinary step on the same handle afterwards still reads the caller's x
    x = prev_labels[cls]
    if precision == "bf16":
        x = wl.from_bf16_bits(wl.to_bf16_bits(x))
    with torch.cuda.stream(gpu.stream):
        compare_step(gpu, ora, x, cls, precision, tol)
    gpu.close()

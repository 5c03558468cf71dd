"""The replica step as one call: steps launched as a CUDA graph (from a plan's 17th on) give bit for bit what the same calls
enqueued one after the other on one stream give, whatever batch they are given, at sizes around the edges of the kernels'
tiles; and the graph keeps the order of the streams, the scalars and the CTA share of the direct calls."""
import threading

import numpy as np
import pytest
import torch

from paper_2003_03477_b200 import synth, trainer

pytestmark = pytest.mark.gpu
DIRECT = 16                                                  # steps a plan enqueues before it builds a graph


def _model(cfg, max_L):
    spec = trainer.ss.MlpSpec(cfg.bottom, cfg.top, cfg.bf16)
    w0 = torch.from_numpy(trainer.pack_params(spec, synth.initial_weights(cfg))).cuda()
    return trainer.Model(cfg.T, cfg.N, cfg.D, cfg.B, cfg.bottom, cfg.top, cfg.bf16, cfg.R, w0, trainer.device_tables(cfg),
                         cfg.lr, cfg.eps, max_L=max_L)


@pytest.mark.parametrize("B,D,bottom,top,bf16", [
    (1, 16, (13, 8), (8,), False), (31, 16, (7, 72), (40,), False), (257, 24, (13, 64), (96, 48), False),
    (700, 64, (16, 256), (256, 256), False),         # 64 x 64 tiles
    (15, 16, (4, 64), (64,), True),                  # fewer samples than a k step
    (33, 16, (1, 8), (24, 16), True), (129, 48, (7, 200, 104), (328, 152), True), (1000, 64, (16, 512), (520, 264), True),
])
def test_repeated_steps_match_the_calls_in_line(B, D, bottom, top, bf16):
    T = 5
    cfg = synth.scaled(synth.CONFIGS["tiny"], R=1, T=T, N=997, D=D, B=B, bottom=bottom + (D,), top=((T + 1) * D,) + top + (1,),
                       bf16=bf16)
    host = [synth.make_batch(cfg, 0, t) for t in range(2)]
    a, b = (_model(cfg, max(x.L for x in host)) for _ in range(2))
    batches = [trainer.DeviceBatch(x.indices, x.offsets, x.dense, x.labels) for x in host]
    torch.cuda.synchronize()
    for t in range(22):                                      # two batches in turn, of different lengths
        a.step(0, batches[t % 2])
    torch.cuda.synchronize()
    for t in range(22):
        b.step(0, batches[t % 2], stream=torch.cuda.default_stream(), overlap_sort=False)
    torch.cuda.synchronize()
    assert a.replicas[0].plan.counts()[:2] == (DIRECT, 22 - DIRECT) and b.replicas[0].plan.counts()[:2] == (22, 0)
    _same(a, b)
    assert np.isfinite(float(a.replicas[0].loss.item())) and not torch.equal(a.tables, trainer.device_tables(cfg))


def _same(a, b):
    assert a.status() == b.status() == 0
    ra, rb = a.replicas[0], b.replicas[0]
    for x, y in ((a.tables, b.tables), (a.row_state, b.row_state), (ra.w, rb.w), (ra.acc, rb.acc), (ra.logit, rb.logit),
                 (ra.loss, rb.loss), (ra.grad_pooled, rb.grad_pooled), (ra.num_unique, rb.num_unique)):
        assert torch.equal(x, y)


def _cfg(B=129, bf16=True, hidden=64):
    return synth.scaled(synth.CONFIGS["tiny"], R=1, T=5, N=997, D=16, B=B, bottom=(13, hidden, 16), top=(96, hidden, 1), bf16=bf16)


def _in_line(model, batch):
    model.step(0, batch, stream=torch.cuda.default_stream(), overlap_sort=False)


@pytest.mark.parametrize("bf16", [False, True])
def test_every_batch_is_launched_as_a_graph(bf16):
    """80 batches of many different lookup counts, each in buffers of its own, then half of them again in fresh ones, with a
    learning rate that changes on the way: all but the first steps are graph launches."""
    cfg = _cfg(bf16=bf16)
    host = [synth.make_batch(cfg, 0, t) for t in range(80)]
    a, b = (_model(cfg, max(x.L for x in host)) for _ in range(2))
    assert len({x.L for x in host}) > 50
    ring = [trainer.DeviceBatch(x.indices, x.offsets, x.dense, x.labels) for x in host]
    torch.cuda.synchronize()
    for t in range(120):
        if t % 8 == 0:
            a.lr = b.lr = 0.01 / (1 + t)
        fresh = ring[t % 80]
        if t >= 80:                                          # freed every time: the allocator hands the memory out again
            x = host[t - 80]
            fresh = trainer.DeviceBatch(x.indices, x.offsets, x.dense, x.labels)
            torch.cuda.synchronize()
        a.step(0, fresh)
        torch.cuda.synchronize()
        _in_line(b, fresh)
        torch.cuda.synchronize()
    direct, launched, updated, graphs = a.replicas[0].plan.counts()
    assert (direct, launched, graphs) == (DIRECT, 120 - DIRECT, 1)
    assert updated > launched                                # other batches: nodes were brought up to date
    _same(a, b)


def test_a_graph_keeps_the_order_of_the_streams():
    """What is on the sort and the MLP stream comes before the step, what comes later on them after it, graph or not."""
    cfg = _cfg()
    x = synth.make_batch(cfg, 0, 0)
    a, b = (_model(cfg, x.L) for _ in range(2))
    batch = trainer.DeviceBatch(x.indices, x.offsets, x.dense, x.labels)
    torch.cuda.synchronize()
    for t in range(DIRECT + 6):
        r = a.replicas[0]
        w = (r.w * (1 + 1e-3 * t)).clone()
        torch.cuda.synchronize()
        with torch.cuda.stream(r.side):
            torch.cuda._sleep(400_000)
            r.num_unique.zero_()                             # the sort writes it
        with torch.cuda.stream(r.mlp):
            torch.cuda._sleep(400_000)
            r.w.copy_(w)
            r.w_bf16.copy_(w)
        a.step(0, batch)
        with torch.cuda.stream(r.mlp):
            after = r.logit.clone()
        b.replicas[0].w.copy_(w)
        b.replicas[0].w_bf16.copy_(w)
        _in_line(b, batch)
        torch.cuda.synchronize()
        assert torch.equal(after, r.logit)
        _same(a, b)
        assert int(r.num_unique.item()) > 0
    assert a.replicas[0].plan.counts()[1] == 6


def test_a_graph_follows_the_cta_share():
    """The tensor-core launches of a graph take as many CTAs as the direct calls would: the number set, and fewer once other
    streams launch such passes too."""
    cfg = _cfg(B=1024, hidden=512)
    x = synth.make_batch(cfg, 0, 0)
    models = [_model(cfg, x.L) for _ in range(3)]
    batch = trainer.DeviceBatch(x.indices, x.offsets, x.dense, x.labels)
    a = models[0].replicas[0].plan
    torch.cuda.synchronize()
    try:
        for t in range(DIRECT + 4):
            models[0].step(0, batch)
        assert a.counts() == (DIRECT, 4, 0, 1)               # the same step: nothing to update
        trainer.ss.ss_mlp_set_flow_ctas(32)
        models[0].step(0, batch)
        assert a.counts()[2] == 2                            # the forward and the backward launch
        trainer.ss.ss_mlp_set_flow_ctas(0)
        models[0].step(0, batch)
        assert a.counts()[2] == 4
        for t in range(4):
            for m in models:
                m.step(0, batch)
        assert a.counts()[2] == 6 and a.counts()[:2] == (DIRECT, 10)
        torch.cuda.synchronize()
        assert models[0].status() == 0
    finally:
        trainer.ss.ss_mlp_set_flow_ctas(0)


def test_plans_of_two_threads_and_of_changing_streams():
    """Two host threads step two models and synchronise the device now and then; one of the models changes between
    overlapped, in-line and caller's streams."""
    cfg = _cfg(bf16=False)
    host = [synth.make_batch(cfg, 0, t) for t in range(3)]
    pairs = [[_model(cfg, max(x.L for x in host)) for _ in range(2)] for _ in range(2)]
    ring = [trainer.DeviceBatch(x.indices, x.offsets, x.dense, x.labels) for x in host]
    other = torch.cuda.Stream()
    torch.cuda.synchronize()
    failed = []

    def train(k):
        try:
            for t in range(90):
                kind = t // 30 if k else 0
                if t % 30 == 0:
                    torch.cuda.synchronize()                 # the streams change
                pairs[k][0].step(0, ring[t % 3], stream=other if kind == 1 else None, overlap_sort=kind != 2)
                if k == 0 and t % 3 == 0:
                    torch.cuda.synchronize()
        except Exception as e:
            failed.append(e)

    threads = [threading.Thread(target=train, args=(k,)) for k in range(2)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    torch.cuda.synchronize()
    assert not failed
    for k in range(2):
        for t in range(90):
            _in_line(pairs[k][1], ring[t % 3])
        torch.cuda.synchronize()
        _same(*pairs[k])
    assert pairs[0][0].replicas[0].plan.counts()[:2] == (DIRECT, 90 - DIRECT)
    assert pairs[1][0].replicas[0].plan.counts()[:2] == (3 * DIRECT, 90 - 3 * DIRECT)

"""Convolutions and weight gradients of different shapes from several host threads at
once, each on a stream of its own: every call succeeds and gives the bits it
gives alone. The shapes of a pair share their kernels and differ in the
shared memory these take (119 and 66 KB, 92 and 62 KB in the convolution)."""
import threading

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_2109_02842_gb300 import build, learned
    build.build()
    learned.lib()
    return learned


def conv_call(L, dims, cin, cout, stream, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = dims[0] * dims[1] * dims[2]
    kp = L.lib().pl_nn_padded_k(cin)
    x = torch.randn((v, cin), device="cuda", generator=g).bfloat16()
    w = torch.zeros((cout, kp), dtype=torch.bfloat16, device="cuda")
    w[:, :27 * cin] = torch.randn((cout, 27 * cin), device="cuda", generator=g) * 0.05
    gy = torch.randn((v, cout), device="cuda", generator=g).bfloat16()
    out = torch.empty((v, cout), device="cuda")
    gw = torch.zeros((cout, kp), device="cuda")
    gb = torch.zeros(cout, device="cuda")
    nbytes = L.lib().pl_nn_wgrad_workspace(*dims, cin, cout)
    work = torch.empty(nbytes // 4, device="cuda")
    handle = L.B._P(stream.cuda_stream)

    def call(clear=True):
        if clear:
            with torch.cuda.stream(stream):
                gw.zero_()
                gb.zero_()
        a = L.lib().pl_nn_conv3d(L._p(x), L._p(w), None, L._p(out), *dims, cin, cout, 0, 0, handle)
        b = L.lib().pl_nn_conv3d_wgrad(L._p(x), L._p(gy), L._p(gw), L._p(gb), L._p(work), nbytes,
                                       *dims, cin, cout, handle)
        return a, b
    return call, (out, gw, gb)


@pytest.mark.parametrize("pair", [(((2, 14, 14), 32, 32), ((3, 2, 4), 32, 32)),
                                  (((3, 300, 1), 16, 64), ((2, 60, 10), 16, 64))])
def test_threads(L, pair):
    jobs = []
    for k in range(4):                # two threads a shape
        dims, cin, cout = pair[k % 2]
        stream = torch.cuda.Stream()
        call, outs = conv_call(L, dims, cin, cout, stream, k)
        torch.cuda.synchronize()
        assert call() == (0, 0)
        stream.synchronize()
        jobs.append((call, stream, outs, [o.clone() for o in outs]))
    torch.cuda.synchronize()
    bad = []
    gate = threading.Barrier(len(jobs))

    def work(call, stream):
        gate.wait()
        for i in range(6000):
            r = call(clear=False)
            if i % 100 == 99:         # (the launch queue never fills)
                stream.synchronize()
            if r != (0, 0) or bad:
                bad.append(r)
                return
    threads = [threading.Thread(target=work, args=j[:2]) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not bad
    for call, _, outs, alone in jobs:
        assert call() == (0, 0)
        torch.cuda.synchronize()
        for o, a in zip(outs, alone):
            assert torch.equal(o, a)

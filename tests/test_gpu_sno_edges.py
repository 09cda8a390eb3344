"""The operator at the edges of its arithmetic, and two operators in two threads."""
import threading

import numpy as np
import pytest

from paper_2209_11922_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _op(N, C, M, L, B, edit=None):
    from paper_2209_11922_gb300.sno import Sno
    w = inputs.SnoWorkload("edges", N=N, C=C, M=M, L=L, window=5, tau=1e-2)
    P = w.init_weights()
    if edit:
        edit(P)
    s = Sno(N, C, M, L, B)
    s.set_params(P)
    u = torch.from_numpy(np.stack([w.u0(i) for i in range(B)]).astype(np.float32)).cuda()
    return s, u, [w.D(i) for i in range(B)]


@pytest.mark.parametrize("C,M", [(16, 12), (32, 24)])
@pytest.mark.parametrize("value", [np.inf, 3e38, 1e20])
def test_activation_of_an_overflowed_value(C, M, value):
    """gelu(+inf) = +inf and gelu(large) = large, in the inference layers as in the training forward: one channel of the last
    layer's bias set to `value`, projected with weight 1 (the other channels are finite and of order 1)."""
    def edit(P):
        P["bp"][0, 3] = value
        P["Wq"][:] = 0.0
        P["Wq"][3] = 1.0
        P["Wp"][0, 3] = 0.0
    s, u, D = _op(32, C, M, 1, 2, edit)
    got = s.forward(u, D).cpu().numpy()
    assert np.all(got == np.float32(value))   # the field's O(1) values are below half an ulp of 1e20
    loss, _ = s.gradient(u, D, u)
    assert loss == np.inf or loss >= float(value) ** 2 * 0.99
    s.close()


def test_operators_of_two_sizes_in_two_threads():
    """Two operators whose launches need different amounts of shared memory, used from two threads on two streams: every call
    succeeds and gives the result it gives alone (no call sets a kernel's limit to its own size, which a launch of the other
    operator would then exceed)."""
    ops = [_op(32, 16, 24, 1, 1), _op(256, 16, 24, 12, 1)]
    want = []
    for s, u, D in ops:
        want.append((s.forward(u, D).clone(), s.gradient(u, D, 0.5 * u)[1]["Wm"].copy()))
    torch.cuda.synchronize()
    errors = []
    go = threading.Barrier(2)

    def work(k):
        s, u, D = ops[k]
        stream = torch.cuda.Stream()
        try:
            go.wait()
            with torch.cuda.stream(stream):
                tgt = 0.5 * u
                for _ in range(1500 if k == 0 else 150):
                    out = s.forward(u, D, stream=stream)
                    _, g = s.gradient(u, D, tgt, stream=stream)
                stream.synchronize()
            assert torch.equal(out, want[k][0]) and np.array_equal(g["Wm"], want[k][1])
        except BaseException as e:   # noqa: BLE001 - reported by the main thread
            errors.append((k, repr(e)))
    ts = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors
    for s, _, _ in ops:
        s.close()

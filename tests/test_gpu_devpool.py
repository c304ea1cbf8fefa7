"""Memory kept from destroyed handles: recycled blocks give the results of fresh ones, from several threads and streams, and
eda_release_cached gives the memory back."""
import threading

import numpy as np
import pytest

from paper_1512_06500_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1512_06500_gb300 import build_lib, eda as E
    build_lib.build()
    E.load()
    return E


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def _run(eda, X, lab, k, cfg, stream=None):
    with eda.build(X, lab, k, cfg, stream=stream) as h:
        V, lam, _, _, code = h.solve(k - 1, 1e-9, stream=stream)
        assert code == 0
    return V, lam


def _problems(eda):
    out = []
    for i, (d, k, nj, prec) in enumerate([(900, 6, 5, eda.EDA_F64), (4100, 12, 7, eda.EDA_F64_TC),
                                          (1200, 30, 10, eda.EDA_F64), (2048, 9, 4, eda.EDA_BF16)]):
        p = synth.gaussian_clusters(d=d, k=k, n_per_class=nj, seed=600 + i)
        out.append((_dev(p.X), _dev(p.labels), k, eda.config(prec=prec, block_b=4, tau=8.0, tc_min_mi=-1)))
    return out


def test_recycled_blocks_give_the_same_bits_and_are_given_back(eda):
    probs = _problems(eda)
    fresh = []
    for pr in probs:
        eda.release_cached()
        fresh.append(_run(eda, *pr))
    eda.release_cached()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    for _ in range(3):
        for pr, (V, lam) in zip(probs, fresh):
            V2, lam2 = _run(eda, *pr)
            assert torch.equal(V, V2) and torch.equal(lam, lam2)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    eda.release_cached()
    # everything but what the caching allocator of the test's own tensors and the driver round up
    assert torch.cuda.mem_get_info()[0] >= before - (64 << 20)


def test_threads_and_streams_share_the_cache(eda):
    probs = _problems(eda)
    want = [_run(eda, *pr) for pr in probs]
    torch.cuda.synchronize()
    bad = []

    def work(first):
        try:
            torch.cuda.set_device(0)
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                for r in range(6):
                    i = (first + r) % len(probs)
                    V, lam = _run(eda, *probs[i], stream=s)
                    s.synchronize()
                    if not (torch.equal(V, want[i][0]) and torch.equal(lam, want[i][1])):
                        bad.append(i)
        except Exception as e:   # noqa: BLE001
            bad.append(e)

    ts = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad, bad

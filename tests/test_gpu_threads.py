"""Host threads that launch the same kernels with different amounts of shared
memory at the same time, each on its own stream: small and bulk calls of the
FP32 coder, of rsc_reconstruct (several sizes of dictionary and code), of
rsc_synthesize (two bases) and of the K-SVD accumulation give what they give
alone, and no launch is refused."""
import ctypes
import threading

import numpy as np
import pytest

from paper_1806_04374_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rsc(cuda_ok):
    import paper_1806_04374_gb300 as rsc
    rsc.load_library()
    return rsc


def _together(calls, rounds=3000):
    """Every call, alone for its result, then all of them at once, a thread
    each; returns what went wrong."""
    import torch
    alone = [[t.clone() for t in f(None)] for f in calls]
    torch.cuda.synchronize()
    wrong = []
    start = threading.Barrier(len(calls))

    def work(i):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                start.wait()
                for _ in range(rounds):
                    got = calls[i](stream)
                stream.synchronize()
                if not all(torch.equal(a, b) for a, b in zip(got, alone[i])):
                    wrong.append((i, "another result"))
        except Exception as e:  # a refused launch
            wrong.append((i, repr(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(calls))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return wrong


def _raw(rsc, fn, out, args):
    """A call of the C ABI into `out`, with little else in a round."""
    import torch
    handles = {}

    def call(stream):
        st = stream or torch.cuda.current_stream()
        a = handles.get(st.cuda_stream)
        if a is None:
            a = handles[st.cuda_stream] = args(out, ctypes.c_void_p(st.cuda_stream))
        status = fn(*a)
        if status != 0:
            raise rsc.RscError(status, fn.__name__)
        return [out]

    return call


def _codes(P, K, M, R):
    import torch
    rng = np.random.default_rng(P + K)
    return {"atom": torch.from_numpy(rng.integers(0, M, (P, K)).astype(np.int32)).cuda(),
            "angle_idx": torch.from_numpy(rng.integers(0, R, (P, K)).astype(np.int32)).cuda(),
            "coef": torch.from_numpy(rng.standard_normal((P, K))).cuda()}


def test_fp32_coder(rsc):
    """16 patches a SM and fewer take blocks of 8 warps, more take 20."""
    import torch
    d = synth.make_dictionary(64, 6, 8, 1)
    x = torch.from_numpy(synth.make_patches(d, 4096, 3, 0.1, 2)[0]).cuda()
    dic = rsc.Dictionary(torch.from_numpy(d).cuda(), 64)
    calls = []
    for n in (32, 2600, 32, 2600):
        xn = x[:n].contiguous()
        out = rsc.encode(dic, xn, 5, "fp32")
        calls.append(lambda s, xn=xn, out=out: list(
            rsc.encode(dic, xn, 5, "fp32", stream=s, out=out).values()))
    assert _together(calls) == []
    dic.close()


def test_way_back(rsc):
    """Blocks of 100, 37 and 1 KB (reconstruct), of 67, 39 and 28 KB
    (synthesize)."""
    import torch
    dics, calls, bases = [], [], []
    vp = ctypes.c_void_p
    lib = rsc.load_library()
    for M, J, kmax, R, K, P in [(8, 4, 16, 128, 16, 40000), (8, 4, 16, 128, 16, 3),
                                (5, 6, 2, 8, 2, 40)]:
        dic = rsc.Dictionary(torch.from_numpy(synth.make_dictionary(M, J, kmax, M)).cuda(), R)
        c = _codes(P, K, M, R)
        dics.append(dic)
        calls.append(_raw(rsc, lib.rsc_reconstruct, rsc.reconstruct(dic, c), lambda o, s, dic=dic, c=c: (
            vp(dic.handle), *c["atom"].shape, vp(c["atom"].data_ptr()), vp(c["angle_idx"].data_ptr()),
            vp(c["coef"].data_ptr()), vp(o.data_ptr()), s)))
    for N, J, kmax, P in [(11, 6, 8, 20000), (11, 6, 8, 30), (3, 1, 1, 20000)]:
        b = rsc.Basis(N, J, kmax)
        c = torch.randn((P, kmax + 1, J, 2), device="cuda")
        bases.append(b)
        calls.append(_raw(rsc, lib.rsc_synthesize, rsc.synthesize(b, c), lambda o, s, b=b, c=c: (
            vp(b.handle), vp(c.data_ptr()), c.shape[0], vp(o.data_ptr()), s)))
    assert _together(calls) == []
    for h in dics + bases:
        h.close()


def test_ksvd(rsc):
    """The residual kernel's blocks of 15 to 80 KB, the covariances' of 207 and
    226."""
    import torch
    dics, calls = [], []
    for M, J, kmax, R, K, P in [(4, 6, 8, 8, 2, 500), (40, 6, 8, 128, 12, 500),
                                (4, 10, 12, 64, 2, 300)]:
        d = synth.make_dictionary(M, J, kmax, M)
        dic = rsc.Dictionary(torch.from_numpy(d).cuda(), R)
        x = torch.from_numpy(synth.make_patches(d, P, 2, 0.1, P)[0]).cuda()
        c = _codes(P, K, M, R)
        dics.append(dic)
        calls.append(lambda s, dic=dic, x=x, c=c: [
            rsc.ksvd_accumulate(dic, x, c, ntop=0, stream=s)[k] for k in ("C", "count")])
    assert _together(calls, 100) == []
    for h in dics:
        h.close()

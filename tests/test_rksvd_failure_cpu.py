"""A device-side error of the R-K-SVD update stops the learning (CPU, the
library's calls replaced): on one rank before the atoms are used or saved, on
two gloo ranks on both of them before anything is summed."""
import os
import socket

import pytest


class _Dic:
    handle = 1

    def __init__(self, d, R):
        self.d = d

    def close(self):
        pass


def _fake(monkeypatch, statuses):
    import torch
    from paper_1806_04374_gb300 import build, rksvd
    build.build()
    d = torch.zeros((2, 1, 3, 2))
    codes = {"resid_norm2": torch.zeros(4)}
    it = iter(statuses)
    monkeypatch.setattr(rksvd, "Dictionary", _Dic)
    monkeypatch.setattr(rksvd, "encode", lambda *a: codes)
    monkeypatch.setattr(rksvd, "ksvd_update", lambda *a: (d + 1, torch.ones(2, dtype=torch.int32)))
    monkeypatch.setattr(rksvd, "device_status", lambda dic: next(it))
    return rksvd, d


def test_learning_stops_before_the_checkpoint(monkeypatch, tmp_path):
    import paper_1806_04374_gb300 as rsc
    ck = str(tmp_path / "c.npz")
    seen = []
    rksvd, d = _fake(monkeypatch, [0, rsc.RSC_ERR_TIMEOUT])
    with pytest.raises(rsc.RscError) as e:
        rksvd.learn(d, d, 4, 1, 3, checkpoint=ck, callback=lambda rec, new: seen.append(rec))
    assert e.value.status == rsc.RSC_ERR_TIMEOUT
    assert len(seen) == 1 and rksvd.load_checkpoint(ck, 4, 1)[1] == 1
    # also in the last coding
    rksvd, d = _fake(monkeypatch, [0, rsc.RSC_ERR_TIMEOUT])
    with pytest.raises(rsc.RscError):
        rksvd.learn(d, d, 4, 1, 1)
    rksvd, d = _fake(monkeypatch, [0, 0])
    assert rksvd.learn(d, d, 4, 1, 1)[2][-1]["iter"] == 1


def _rank(rank, world, port, q):
    import torch
    import torch.distributed as dist
    os.environ.update(MASTER_ADDR="127.0.0.1", MASTER_PORT=str(port))
    dist.init_process_group("gloo", rank=rank, world_size=world)
    import paper_1806_04374_gb300 as rsc
    from paper_1806_04374_gb300 import rksvd
    acc = {"C": torch.full((2, 3, 3), 1.0, dtype=torch.float64),
           "count": torch.full((2,), rank + 1, dtype=torch.int32),
           "top_err": torch.zeros(1), "top_idx": torch.zeros(1, dtype=torch.int64),
           "top_vec": torch.zeros((1, 1, 3, 2))}
    finished = []
    rksvd.ksvd_accumulate = lambda *a: acc
    rksvd.ksvd_finish = lambda dic, C, cnt, *a: finished.append((float(C[0, 0, 0]), cnt.tolist()))
    out = []
    for status in (0, rsc.RSC_ERR_TIMEOUT if rank == 1 else 0):
        rksvd.device_status = lambda dic: status
        try:
            rksvd.update_distributed(None, torch.zeros(1), None, dist.group.WORLD)
            out.append(0)
        except rsc.RscError as e:
            out.append(e.status)
    q.put((rank, out, finished, float(acc["C"][0, 0, 0])))
    dist.destroy_process_group()


def test_every_rank_stops():
    import torch.multiprocessing as mp
    import paper_1806_04374_gb300 as rsc
    from paper_1806_04374_gb300 import build
    build.build()
    with socket.socket() as s:
        s.bind(("127.0.0.1", 0))
        port = s.getsockname()[1]
    ctx = mp.get_context("spawn")
    q = ctx.Queue()
    procs = [ctx.Process(target=_rank, args=(r, 2, port, q)) for r in range(2)]
    for p in procs:
        p.start()
    res = sorted(q.get(timeout=180) for _ in procs)
    for p in procs:
        p.join(timeout=60)
        assert p.exitcode == 0
    for _, out, finished, c in res:
        assert out == [0, rsc.RSC_ERR_TIMEOUT]
        assert finished == [(2.0, [3, 3])]  # the first update, not the second
        assert c == 2.0                     # nothing summed in the second

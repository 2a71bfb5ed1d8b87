"""The host-buffer entry point from several threads at once, each with its own buffers and stream: the copy streams and events
behind it are shared, and one call's waits must not take another's records."""
import threading

import pytest
import torch

import paper_2607_14568_b200 as gdn
from workloads import get_config, make_inputs

pytestmark = pytest.mark.gpu


def _host(a):
    import numpy as np
    t = torch.from_numpy(a.view(np.int16)).view(torch.bfloat16) if a.dtype == np.uint16 else torch.from_numpy(a)
    return t.pin_memory()


def test_calls_of_several_threads_keep_apart():
    gdn.gdn_set_workspace(None)                            # calls on different streams may not share scratch
    jobs = []
    for i, T in enumerate((4096, 6144 + 100, 4096 + 1, 10240)):      # two to five pieces
        x = make_inputs(get_config("long", T=T, H=2, seed=100 + i))
        h = {n: _host(getattr(x, n)) for n in ("q", "k", "v", "log_alpha", "beta", "initial_state")}
        jobs.append((h, torch.empty(h["v"].shape, dtype=torch.bfloat16, pin_memory=True),
                     torch.empty(1, 2, 128, 128, pin_memory=True),
                     torch.empty(gdn.gdn_host_staging_bytes(1, T, 2, 128, 128), dtype=torch.uint8, device="cuda"), torch.cuda.Stream()))

    def call(job):
        h, out, fin, staging, stream = job
        gdn.gdn_chunk_prefill_host(h["q"], h["k"], h["v"], h["log_alpha"], h["beta"], h["initial_state"], out, fin, None, staging, stream=stream)

    want = []
    for job in jobs:
        call(job)
        torch.cuda.synchronize()
        want.append((job[1].clone(), job[2].clone()))
    for _ in range(5):
        for job in jobs:
            job[1].zero_(); job[2].zero_()
        go = threading.Barrier(len(jobs))
        failed = []

        def run(job):
            try:
                go.wait(timeout=30)
                for _ in range(3):
                    call(job)
                job[4].synchronize()
            except Exception as e:  # noqa: BLE001 - reported by the main thread
                failed.append(e)

        ts = [threading.Thread(target=run, args=(job,)) for job in jobs]
        for t in ts: t.start()
        for t in ts: t.join()
        assert not failed, failed
        assert gdn.gdn_query_status() == 0
        for job, (o, f) in zip(jobs, want):
            assert torch.equal(job[1], o) and torch.equal(job[2], f)

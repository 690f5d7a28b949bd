"""What a launch keeps from the driver (CTAs per SM, the shared-memory limit) is
kept per device and is safe between threads: the cache alone on the host, and two
threads applying patterns of different chunk lengths on the GPU (each with more
than 48 KB of shared memory, so a limit lowered by one would refuse the other)."""
from __future__ import annotations

import os
import subprocess
import threading

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_cache_per_device_and_thread(tmp_path):
    exe = tmp_path / "launch_cache"
    inc = os.path.join(HERE, "..", "paper_1703_01325_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O2", "-pthread", "-I", inc, os.path.join(HERE, "launch_cache_main.cpp"),
                    "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


@pytest.mark.gpu
def test_two_threads_two_chunk_lengths(libbilu):
    torch = pytest.importorskip("torch")
    import paper_1703_01325_gb300.bilu as B
    from paper_1703_01325_gb300.reservoir import reservoir_system
    torch.cuda.set_device(0)
    b = 8
    S = reservoir_system(40, 16, 4, b, sigma=1.0, accum=0.01, seed=3)
    vals, rhs = (torch.from_numpy(np.ascontiguousarray(a).reshape(-1)).cuda() for a in (S.vals, S.rhs))
    jobs = []
    old = B.bilu_get_trisolve_chunk()
    try:
        for rows in (680, 1024):  # 52 and 78 KB per CTA
            B.bilu_set_trisolve_chunk(rows)
            P = B.bilu_symbolic(S.n, S.row_ptr, S.col_idx, 0).upload()
            F, _ = B.bilu_factor(P, b, vals)
            jobs.append((P, F, B.bilu_apply(P, b, F, rhs)))
    finally:
        B.bilu_set_trisolve_chunk(old)
    torch.cuda.synchronize()
    failed = []

    def work(P, F, want):
        torch.cuda.set_device(0)
        s = torch.cuda.Stream()
        x, w = torch.empty_like(rhs), B.workspace(P.apply_workspace_bytes(b))
        torch.cuda.synchronize()
        try:
            for _ in range(300):
                B.bilu_apply(P, b, F, rhs, x=x, work=w, stream=s)
            s.synchronize()
            if not torch.equal(x, want):
                failed.append("values")
        except Exception as e:  # noqa: BLE001 - reported by the test
            failed.append(repr(e))

    ts = [threading.Thread(target=work, args=j) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not failed, failed

"""Handles used from several host threads at once, a stream each: their launches
differ in shared memory and must not undo each other's settings."""

import ctypes
import threading

import pytest
import torch

from workloads.synth import Workload, make_inputs

pytestmark = pytest.mark.gpu


def test_cluster_kernel_from_several_threads(monkeypatch):
    import paper_2505_12398_gb300 as tv
    w = Workload("threads", 2, 8008, levels=(2, 3), branching=(2, 2), sigma=1.0)
    inp = make_inputs(w, seed=1, device="cuda")
    B, R = inp.parents.shape
    handles = []
    for shape in ("8,1,0", "8,1,2") * 3:     # the ring as large as fits, and two stages
        monkeypatch.setenv("TV_FUSED_PLAN", shape)
        handles.append(tv.Verifier(8008, R - 1, B, "bf16", path="cluster"))
    want = handles[0].verify(inp.parents, inp.tokens, inp.logits, inp.draft_probs,
                             inp.temperature, inp.uniforms)
    torch.cuda.synchronize()
    wrong = []

    def work(v):
        stream = torch.cuda.Stream()
        out = [torch.empty_like(x) for x in want]
        ptr = [ctypes.c_void_p(x.data_ptr()) for x in
               (inp.parents, inp.tokens, inp.logits, inp.draft_probs, inp.uniforms, *out)]
        call = v.lib.tv_verify_batch
        stream.wait_stream(torch.cuda.default_stream())
        for _ in range(3000):
            rc = call(v.handle, B, R - 1, *ptr[:4], inp.temperature, *ptr[4:],
                      ctypes.c_void_p(stream.cuda_stream))
            if rc != 0:
                wrong.append(rc)
                break
        stream.synchronize()
        if not all(torch.equal(x, y) for x, y in zip(out, want)):
            wrong.append("results")

    threads = [threading.Thread(target=work, args=(v,)) for v in handles]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for v in handles:
        assert v.status() & ~16 == 0
        v.close()
    assert not wrong, wrong

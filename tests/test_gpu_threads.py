"""Contexts of different layer counts used by two threads at once, each on a stream of its own: the
kernels' shared-memory grants follow from the layers and are shared by all contexts of a device."""
import threading

import numpy as np
import pytest

import paper_2607_24141_gb300 as pz
from tiny import tiny_problem

pytestmark = pytest.mark.gpu


def test_two_threads_with_different_layer_counts():
    import torch
    probs = [tiny_problem(n_lambda=400, n_depth=nd, n_lines=80, W=90) for nd in (128, 9)]
    precs = (pz.PZ_MIXED, pz.PZ_FP64)

    def run(prob, prec, stream, reps, out):
        with torch.cuda.stream(stream):
            s = pz.Synthesizer(prob, prec)
            dL = torch.ones(s.n_out, dtype=torch.float32, device=s.device)
            g = [torch.empty(s.n_lines, dtype=torch.float32, device=s.device) for _ in range(2)]
            for _ in range(reps):
                f = s.forward()
                s.backward(dL, *g)
            stream.synchronize()
            out.append([f.cpu().numpy()] + [x.cpu().numpy() for x in g])
            s.close()

    for prec in precs:
        got = [[], []]
        threads = [threading.Thread(target=run, args=(p, prec, torch.cuda.Stream(), 30, got[k]))
                   for k, p in enumerate(probs)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        for k, p in enumerate(probs):
            want = []
            run(p, prec, torch.cuda.current_stream(), 1, want)
            assert len(got[k]) == 1
            for a, b in zip(got[k][0], want[0]):
                assert np.all(np.isfinite(a)) and np.max(np.abs(a - b)) <= 2e-6 * np.max(np.abs(b))

"""Kernels launched while the one before them still runs, inside whole calls: training steps (single network and
per-species ensemble, plain and dependent launches mixed), the forward pass and the learned step with its
fallback and properties, at batches and cell counts on both sides of the rule. Each result has the bits of the same
calls in a process whose launches all wait for their end (CUDA_LAUNCH_BLOCKING), and the learned step replayed from
a CUDA graph those of the direct call."""
import hashlib
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _digest(*arrays):
    h = hashlib.sha256()
    for a in arrays:
        h.update(a if isinstance(a, bytes) else a.tobytes())
    return h.hexdigest()[:16]


def work(repeat):
    """name -> digests of `repeat` runs, none synchronised before its end."""
    import numpy as np
    import torch
    from paper_2312_05800_gb300 import binding, synth
    out = {}
    m = synth.get_mech("c2")
    dm = binding.Mech(m)
    n = 40000
    ld = synth.padded_ld(n)
    T, p, Y = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in synth.states_profiles(m, n, 17, ld))
    Y1 = Y * (1.0 + 1e-3 * torch.sin(torch.arange(Y.numel(), device="cuda", dtype=torch.float64).reshape(Y.shape)))

    def net(ensemble=False, **kw):
        a = binding.Mlp(dm, hidden=(104, 56, 24) if ensemble else (1600, 800, 400), dt=1e-6, seed=5, ensemble=ensemble, **kw)
        binding.chem_mlp_fit_norm(a, n, ld, T, p, Y, Y1)
        return a

    for ensemble in (False, True):
        for batch in (8, 264, 4096):
            for r in range(repeat):
                a = net(ensemble, chunk=4096, max_batch=4096)
                loss = torch.zeros(4, 4, device="cuda")
                for k in range(4):
                    binding.mlp_train_step(a, batch, None, ld, T, p, Y, Y1, 1e-3, loss[k] if k % 2 == 0 else None)
                torch.cuda.synchronize()
                out.setdefault("train %d %d" % (ensemble, batch), []).append(
                    _digest(a.get_params(), a.get_grads(), loss.cpu().numpy()))
                a.free()
    a = net(chunk=32768)
    binding.chem_mlp_fit_ood_multi(a, dm, 20000, ld, T, p, Y, [m.roles["oxidizer"], m.roles["co2"]], nbins=16, min_count=1)
    opts = binding.make_opts(rtol=1e-2, atol_Y=1e-8, atol_T=1e-2, h0=1e-9, mode=binding.CHEM_ODE_MIXED)
    for cells in (300, 2500, n):
        u = torch.zeros(cells, 32, device="cuda")
        for r in range(repeat):
            binding.chem_mlp_forward(a, cells, ld, T, p, Y, u, 32)
            torch.cuda.synchronize()
            out.setdefault("forward %d" % cells, []).append(_digest(u.cpu().numpy()))
        S, st = torch.zeros(m.N + 1, ld, dtype=torch.float64, device="cuda"), torch.zeros(ld, dtype=torch.int32, device="cuda")
        props = torch.zeros(4 + m.N, ld, device="cuda")

        def step():
            S[0].copy_(T)
            S[1:].copy_(Y)
            for _ in range(2):
                binding.chem_step_ann_props(dm, a, cells, ld, 1e-6, binding.CHEM_PREC_BF16, opts, S[0], p, S[1:], st,
                                            props[0], props[1], props[2], props[3], props[4:])

        def result():
            torch.cuda.synchronize()
            return _digest(S.cpu().numpy(), st.cpu().numpy(), props.cpu().numpy())

        for r in range(repeat):
            step()
            out.setdefault("step %d" % cells, []).append(result())
        if repeat > 1:
            graph = torch.cuda.CUDAGraph()
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                step()
            torch.cuda.current_stream().wait_stream(side)
            with torch.cuda.graph(graph):
                step()
            for r in range(repeat):
                S.zero_()
                props.zero_()
                graph.replay()
                out["step %d" % cells].append(result())
    return out


def _child(repeat, **env):
    code = "import json, sys; sys.path[:0] = [%r]; from tests.test_gpu_dependent_steps import work; print('RESULT ' + json.dumps(work(%d)))" % (ROOT, repeat)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, cwd=ROOT, timeout=600,
                       env=dict(os.environ, **env))
    assert r.returncode == 0 and "RESULT " in r.stdout, r.stdout + r.stderr[-4000:]
    import json
    return json.loads(r.stdout.split("RESULT ")[1])


def test_whole_calls_have_the_bits_of_serial_launches():
    want, got = _child(1, CUDA_LAUNCH_BLOCKING="1"), _child(3)
    assert want.keys() == got.keys() and len(want) == 12
    for name, (digest,) in want.items():
        assert set(got[name]) == {digest}, name
    assert len(got["step 300"]) == 6

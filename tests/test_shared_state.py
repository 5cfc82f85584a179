"""One context per host thread: no call may stage its launch in memory that calls on other contexts share."""
import glob
import os
import re

import numpy as np
import pytest

import workloads

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0906_2569_gb300", "csrc")


def test_no_process_wide_mutable_state():
    """Variables of static storage inside functions are constant, one per thread, or atomic (static check of csrc/)."""
    variable = re.compile(r"^\s+static\s+(?!constexpr\b|const\b|thread_local\b|std::atomic\b|__)"
                          r"[\w:]+(?:<[^;()]*>)?[\s*&]+\w+(?:\[[^\]]*\])*\s*(?:=[^;]*|\{[^;]*\})?;", re.M)
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*"))):
        text = open(path).read()
        found += [f"{os.path.basename(path)}: {m.group(0).strip()}" for m in variable.finditer(text)]
    assert not found, found


def test_shared_memory_limits_are_set_once_per_device():
    """The limit belongs to the device's kernel, not to a context: a call that set it to its own size could lower it
    between another thread's set and launch."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*"))):
        for line in open(path):
            if "cudaFuncAttributeMaxDynamicSharedMemorySize" in line:
                assert "smem_optin" in line, f"{os.path.basename(path)}: {line.strip()}"


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [0, 1])
def test_threads_with_contexts_of_their_own(lib, precision):
    """Four threads apply H of different boxes, block sizes and projector counts at once, each on its own context and stream;
    every result equals that of the same context used alone."""
    import threading
    import torch
    from paper_0906_2569_gb300 import binding as B
    cases = [(8.0, 10.0, 2, 5), (10.0, 12.0, 3, 17), (12.0, 9.0, 8, 9), (9.0, 20.0, 5, 12)]
    jobs = []
    for i, (a, ecut, nat, nb) in enumerate(cases):
        lat = np.diag([a, a, a])
        m = B.hpsi_gsphere(lat, ecut, np.zeros(3))
        n = workloads.cubic_box(a, ecut)
        rng = np.random.default_rng(i)
        atoms = rng.random((nat, 3)) @ lat
        vr = rng.standard_normal((n, n, n))
        beta = workloads.beta(lat, atoms, np.zeros(3), m)
        stream = torch.cuda.Stream()
        ctx = B.hpsi_setup(lat, ecut, [np.zeros(3)], (n, n, n), vr, [beta], workloads.dmat(nat), precision,
                           stream.cuda_stream)
        B.hpsi_set_option(ctx, B.HPSI_OPT_AUTOTUNE, 0)
        with torch.cuda.stream(stream):
            x = torch.from_numpy(workloads.random_block(len(m), nb, i)).cuda()
            half = x[:, len(m) // 2:].contiguous()
            half[:, 0].imag.zero_()
            alone = [torch.empty_like(x), torch.empty_like(x), torch.empty_like(half)]
            stream.synchronize()
            B.hpsi_apply(ctx, 0, x, alone[0])
            B.hpsi_apply_batch(ctx, [0], [x], [alone[1]])
            B.hpsi_apply_gamma(ctx, 0, half, alone[2])
        B.hpsi_sync(ctx)
        jobs.append((ctx, stream, x, half, alone))
    wrong = []
    start = threading.Barrier(len(jobs))

    def work(i):
        ctx, stream, x, half, alone = jobs[i]
        try:
            with torch.cuda.stream(stream):
                out = [torch.empty_like(t) for t in alone]
                start.wait()
                for it in range(50):
                    for t in out:
                        t.fill_(float("nan"))
                    B.hpsi_apply(ctx, 0, x, out[0])
                    # a new output each time is a new argument list: run, then captured
                    y = torch.empty_like(x) if it % 2 else out[1]
                    B.hpsi_apply_batch(ctx, [0], [x], [y])
                    B.hpsi_apply_gamma(ctx, 0, half, out[2])
                    B.hpsi_sync(ctx)
                    if not (torch.equal(out[0], alone[0]) and torch.equal(y, alone[1]) and torch.equal(out[2], alone[2])):
                        wrong.append((i, it))
        except Exception as e:   # reported by the main thread
            wrong.append((i, repr(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for ctx, *_ in jobs:
        ctx.close()
    assert not wrong, wrong[:5]

"""Instances of a cohort that end their solves in different iterations.

A solve ends inside the x/r update (p.q <= 0) or the p update (tolerance, cap,
r.z <= 0): block 0 of the instance raises its done flag while other blocks of
the same launch may still be starting.  Blocks of these two steps pass barriers
behind their test of the flag, so a block has to leave as a whole or not at all.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2505_13390_gb300", "csrc")


def _expand(body, macros):
    for name, text in macros.items():
        body = re.sub(rf"\b{name}\b", lambda _: text, body)
    return body


def test_ending_steps_read_the_flag_once_per_block():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "solve.cu")).read())
    macros = {n: t.replace("\\\n", "\n")
              for n, t in re.findall(r"#define (COHORT_\w+)[ \t]*\\\n((?:[^\n]*\\\n)*[^\n]*)", src)}
    ending = 0
    for name, body in re.findall(r"__global__ void (kb_\w+)\([^)]*\) \{\n(.*?)\n\}", src, re.S):
        if not re.search(r"\b(xr_update_body|p_update_body)\b", body):
            continue
        ending += 1
        reads = re.findall(r"if \(([^;]*is_done[^;]*)\) return;", _expand(body, macros))
        assert reads and all("__syncthreads_or(threadIdx.x == 0 &&" in r for r in reads), name
    assert ending == 2


@pytest.mark.gpu
def test_members_that_end_apart_equal_alone():
    """Caps of 1 to 30 iterations, tolerances from 1e-1 to 1e-6 and an
    indefinite A (negative compliance) side by side: every status, iteration
    count and state is that of the instance served alone."""
    import numpy as np
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_13390_gb300.meshgen import cloth, default_params, hex_block
    from paper_2505_13390_gb300.mgpbd import Batch
    common = dict(precision=1, level0_op=1, use_graphs=1, max_iter=2, setup_interval=2, coarse_max=40)
    ms = []
    for k, (cap, rtol) in enumerate([(1, 1e-6), (7, 1e-6), (8, 1e-6), (9, 1e-6), (30, 1e-6),
                                     (5000, 1e-1), (5000, 1e-3), (5000, 1e-6)]):
        mesh = (cloth(20 + 9 * k, plane="xz", alpha=1e-6, pin="corners", seed=k) if k % 2 else
                hex_block(5 + k, 6, 7, h=0.01, alpha=1e-7, pin="x0", seed=k))
        ms.append((mesh, default_params(pcg_maxiter=cap, pcg_rtol=rtol, **common)))
    ms.append((hex_block(8, 6, 7, h=0.01, alpha=-1e-9, pin="x0", seed=9),
               default_params(pcg_maxiter=500, **common)))

    def serve(cohort, active):
        b = Batch(64 << 30, active, cohort=cohort)
        ids = [b.add(m, p) for m, p in ms]
        _, res = b.run([(k, i, 1, 0.0) for k, i in enumerate(ids)])
        states = [b.state(i) for i in ids]
        b.close()
        return sorted((r["id"], r["status"], r["pcg_iters"]) for r in res), states

    alone, s1 = serve(False, 1)
    mixed, s2 = serve(True, len(ms))
    assert alone == mixed
    for (x1, v1), (x2, v2) in zip(s1, s2):
        assert np.array_equal(x1, x2) and np.array_equal(v1, v2)

"""The elementary functions that the accuracy tests run (csrc/trig.cuh) are the
ones that the kernels call: one definition each in the device sources, and the
step and the noise call it.  On the GPU, the normals of the noise stream are
within the error of those functions."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_05773_gb300", "csrc")


def _sources():
    return {os.path.basename(p): open(p).read() for p in glob.glob(os.path.join(CSRC, "*.cuh"))}


def test_one_definition_of_each_function():
    src = _sources()
    for constant in ("2.7557318844628753e-06f",  # sin's series
                     "0.636619746685028f), T(12582912.0f)",  # the quadrant
                     "0.01227184630308513f", "1.6525916589735634e-07f"):  # the noise's angle, ln 2
        assert [n for n in src if constant in src[n]] == ["trig.cuh"], constant
        assert src["trig.cuh"].count(constant) == 1, constant


def test_the_kernels_call_them():
    src = _sources()
    assert len(re.findall(r"\bbox_muller<NS>\(", src["rollout.cuh"])) == 2
    assert len(re.findall(r"\bbox_muller<1>\(", src["rollout.cuh"])) == 2
    assert len(re.findall(r"\bstate_sincos\(", src["rollout.cuh"])) >= 5
    scalar = src["trig.cuh"][src["trig.cuh"].index("inline float neg2_log_unit"):]
    assert scalar.count("box_muller<1, true>(") == 2


@pytest.mark.gpu
@pytest.mark.parametrize("seed,counter", [(3, 1), (2**63 + 5, 77)])
def test_normals_within_the_functions_error(seed, counter):
    """n = r (cos, sin) with r = sqrt(-2 ln u_a).  In units of 2^-23 r: the
    logarithm is within 1.42 ulp of -2 ln u_a, at most 1.42 2^-23 of it, and its
    root halves that (0.71); the root by one Newton step 0.6 ulp; cos and sin
    0.51 ulp of 1; the product half an ulp (0.5): 2.32 in all."""
    import numpy as np
    import torch
    import oracle
    from paper_2508_05773_gb300 import build as native_build
    native_build.build()
    import paper_2508_05773_gb300 as pkg
    n_samples, H, n_blocks = 2000, 50, 10
    normals = torch.empty((n_samples, H, n_blocks, 4), dtype=torch.float32, device="cuda")
    assert pkg.brmppi_noise_blocks(seed, counter, n_samples, H, n_blocks, None, normals) == 0
    torch.cuda.synchronize()
    gn = normals.cpu().numpy().astype(np.float64)
    _, on = oracle.noise_table(seed, counter, n_samples, H, n_blocks)
    r = np.repeat(np.hypot(on[..., 0::2], on[..., 1::2]), 2, axis=-1)
    worst = float(np.max(np.abs(gn - on) / r) * 2.0**23)
    assert worst <= 2.32, worst

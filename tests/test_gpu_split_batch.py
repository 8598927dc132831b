"""A batch of split-form models follows the arithmetic of each model's own run, whatever the spins in it: a != 0 takes
the Kerr-Schild point form of the FP64 geodesic and a = 0 the component form, superphoton by superphoton.
The form truncates FP64 components to FP32, so two FP64 geodesics that differ in their last bits show as
6e-8 in a weight now and then; with some 10^6 superphotons of many scatterings that moves a bin by far more
than the 1e-11 left to the order of its sum."""
import numpy as np
import pytest

from helpers import requires_gpu
from paper_2602_13198_gb300 import mc, synth

pytestmark = [pytest.mark.gpu, requires_gpu]


def run_both(specs, weights=None):
    def model(p, g):
        m = mc.Model(p, device=0, precision="split", surrogate=weights is not None)
        m.set_grid(g)
        if weights is not None:
            m.surrogate_weights(weights)
        return m

    ns, seeds = [n for _, n in specs], [40 + i for i in range(len(specs))]
    own = []
    for ((p, g), n_s), sd in zip(specs, seeds):
        m = model(p, g)
        own.append((m.run(n_s, sd), m.spectrum_sums().copy()))
    batch = [model(p, g) for (p, g), _ in specs]
    st = mc.run_batch(batch, ns, seeds)
    for k in ("n_emit", "n_child", "n_rec", "n_abs", "n_capt", "n_steps", "n_events"):
        assert st[k] == sum(r[0][k] for r in own), k
    for m, (_, ref) in zip(batch, own):
        s = m.spectrum_sums()
        assert np.array_equal(s[..., 2], ref[..., 2])
        assert np.allclose(s[..., :2], ref[..., :2], rtol=1e-11, atol=0)


def test_split_batch_follows_each_models_own_run():
    run_both([(synth.torus(a=0.9375, n1=128, n2=64, R_high=1.0, seed=1), 1e6),
              (synth.torus(a=-0.94, n1=97, n2=49, R_high=1.0, kappa=4.5, brems=1, seed=2), 3e5),
              (synth.torus(a=0.0, n1=96, n2=48, R_high=1.0, seed=3), 3e5),
              (synth.torus(a=0.5, n1=48, n2=24, n3=16, R_high=10.0, dtype=np.float32, seed=4), 3e5)])


def test_split_batch_with_network_follows_each_models_own_run():
    rng = np.random.default_rng(11)
    w = [rng.normal(0, 1.0, (64, 3)), rng.normal(0, 0.5, 64), rng.normal(0, 0.15, (64, 64)), rng.normal(0, 0.2, 64),
         rng.normal(0, 0.02, (3, 64)), np.array([-0.5, 0.3, 0.0])]
    run_both([(synth.torus(a=0.9375, n1=128, n2=64, R_high=10.0, seed=5), 3e5),
              (synth.torus(a=0.0, n1=96, n2=48, R_high=10.0, seed=6), 2e5)],
             np.concatenate([v.ravel() for v in w]).astype(np.float32))

"""The filter's default launch variant against the plain form of the same block
shape (NT x PPT): the same arithmetic on more resident warps, so the states are
equal bit for bit, at the edges of each block size."""
import numpy as np
import pytest
import torch

from synth import preset

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2505_08222_gb300 as ut  # noqa: E402


@pytest.mark.parametrize("ess", [0, 8])
@pytest.mark.parametrize("P", [1, 31, 128, 129, 256, 257, 512, 1000, 1025, 2048])
def test_default_variant_gives_the_plain_forms_bits(P, ess):
    p = preset("fleet5", n_envs=9).replace(n_particles=P, d_model=0, pf_ess_num=ess)
    act = torch.from_numpy(np.random.default_rng(P).integers(0, 7, 45).astype(np.int32)).cuda()
    got = []
    for plain in (False, True):
        env = ut.Env(p)
        env.reset(3)
        name = env.pf_variant_name()
        if plain:
            labels = {ut.lib.pf_variant_label(v).decode(): v for v in env.pf_variants()}
            base = name.split("m")[0]
            assert base in labels and name != base
            env.set_pf_variant(labels[base])
        for _ in range(4):
            env.step(act)
        st = env.state()
        got.append([st[k].clone() for k in ("px", "py", "pvx", "pvy", "estx", "esty")])
    for a, b in zip(*got):
        assert torch.equal(a, b)

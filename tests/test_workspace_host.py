"""Workspaces stay within the sizes that callers have laid arenas out for (no GPU)."""

import pytest

# np, nc, pos_bytes, lowmem (20 steps, default pk_mesh_max): bytes
SIZES = [(32, 16, 1, False, 5153536), (32, 16, 1, True, 4875008), (32, 16, 2, False, 5350144),
         (64, 32, 1, False, 40776192), (64, 32, 1, True, 38547968), (64, 64, 1, False, 303683840),
         (64, 64, 2, False, 305256704), (128, 64, 1, False, 325703936), (128, 64, 1, True, 307878144),
         (256, 128, 1, False, 2604945664), (256, 128, 1, True, 2462339328), (256, 128, 2, False, 2705608960),
         (512, 256, 1, False, 11174530816), (512, 256, 1, True, 4664970496), (512, 512, 1, True, 21209899776),
         (2048, 1024, 1, True, 264155308800)]


@pytest.mark.parametrize("np_,nc,pos_bytes,lowmem,most", SIZES)
def test_workspace_is_no_larger(np_, nc, pos_bytes, lowmem, most):
    from paper_2003_03931_gb300 import build
    from paper_2003_03931_gb300.sim import SimConfig, workspace_bytes
    build.build()
    got = workspace_bytes(SimConfig(np=np_, nc=nc, n_steps=20, pos_bytes=pos_bytes, lowmem=lowmem))
    assert most - (8 << 20) < got <= most

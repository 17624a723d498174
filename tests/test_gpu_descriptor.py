"""The step descriptor and the commit lengths reach the device by value (up to 32 sequences) or by a copy (more): the same
sequences decoded in one batch of 40 and in two of 20 must give the same tokens and the same records."""
import numpy as np
import pytest
import torch

import lsp_synth as S
from gpu_util import DEV

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("topology,lagged", [(0, 0), (0, 1), (1, 0)])
def test_batches_on_both_sides_of_the_inline_descriptor(topology, lagged):
    from paper_2603_05454_b200 import LSPDecoder, SchedCfg
    sh = S.ModelShape(2, 256, 4, 2, 64, 512, 1024, dtype="fp32", head_scale=1.5, w_std=0.0625)
    w = S.make_weights(sh, 0, device=DEV)
    B, P, G = 40, 9, 11
    prompt = S.make_prompt(B, P, sh, 3).to(DEV)
    bm = S.delimiter_bitmap(sh.vocab, 1, 64).to(DEV)
    sched = SchedCfg(tau=0.05, delim_bitmap=bm, topology=topology, mode=2 if topology else 0, fixed_k=3)
    gen = [G - b % 5 for b in range(B)]
    out = {}
    for lo, hi in ((0, 40), (0, 20), (20, 40)):
        dec = LSPDecoder(sh, w, sched, hi - lo, P + G, device=DEV)
        dec.set_option(4, lagged)
        tokens = torch.zeros(hi - lo, P + G, dtype=torch.int32, device=DEV)
        tokens[:, :P] = prompt[lo:hi]
        dec.begin(tokens, [P] * (hi - lo), gen[lo:hi])
        n, recs = dec.generate(max_recs=(hi - lo) * (G + 1))
        per = [[tuple(r[k] for k in ("n_before", "rows", "L_run", "L_commit", "flags", "flips", "flip_base")) for r in recs[b::hi - lo] if r["n_before"]]
               for b in range(hi - lo)]
        out[lo, hi] = (tokens.cpu().numpy(), per)
        dec.close()
    whole = out[0, 40]
    halves = (np.concatenate([out[0, 20][0], out[20, 40][0]]), out[0, 20][1] + out[20, 40][1])
    assert np.array_equal(whole[0], halves[0])
    assert whole[1] == halves[1]

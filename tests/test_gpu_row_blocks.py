"""GPU parity of dense and grouped linears on small, ragged shapes: with the kernels that the library picks, and with other
families, tile widths and K splits forced.

The library reads its knobs (DPS_FORCE_PATH, DPS_FORCE_SPLIT, DPS_PAIR_TOKENS, DPS_PAIR_SPLIT) once per process, so each
forced run is a child process: this file executed as a script compares against the oracle and prints one line per case.
"""
import os
import subprocess
import sys

import pytest

REPO = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _cases():
    import numpy as np
    import torch

    import oracle
    import paper_2609_34380_b200 as dps
    from paper_2609_34380_b200 import workloads
    from tests.helpers import assert_close_to_oracle, split_both, to_np_words

    dev = "cuda:0"
    # dense: N not a multiple of 256 (a pair's second row block ragged or absent), K with a ragged last block,
    # token counts that leave a partial last token tile
    for (N, K, M) in [(640, 1088, 200), (128, 512, 65), (904, 2064, 300), (392, 272, 577)]:
        for forced_enc in (dps.DPS_ENC_AUTO, dps.DPS_ENC_E5M2):
            w = workloads.weights(N, K, 11 + N, device=dev)
            p, r, enc, p_ref, r_ref = split_both(w, forced_enc, dev)
            x = workloads.activations(M, K, 13 + M, device=dev)
            for mode in (dps.DPS_MODE_FAST, dps.DPS_MODE_FULL):
                y = dps.dps_linear(mode, enc, x, p, r if mode else None)
                ref = oracle.linear(mode, enc, to_np_words(x), p_ref, r_ref, threads=8)
                assert_close_to_oracle(y, ref, f"dense N={N} K={K} M={M} enc={enc} mode={mode}")
                print(f"ok dense N={N} K={K} M={M} enc={enc} mode={mode}")
    # grouped: experts with 0, few and more than one tile of rows; N ragged against 256; 45 and 100 rows per expert, on the
    # tiles of one CTA and on CTA pairs
    for (E, N, K, T) in [(4, 384, 1040, 90), (3, 136, 528, 150)]:
        ps, rs, encs, p_refs, r_refs = [], [], [], [], []
        for e in range(E):
            w = workloads.weights(N, K, 50 + e, device=dev)
            if e == 1:
                w = workloads.with_outlier(w)
            p, r, enc, p_ref, r_ref = split_both(w, dps.DPS_ENC_AUTO, dev)
            ps.append(p), rs.append(r), encs.append(enc), p_refs.append(p_ref), r_refs.append(r_ref)
        p, r = torch.stack(ps), torch.stack(rs)
        p_ref, r_ref = np.stack(p_refs), np.stack(r_refs)
        x = workloads.activations(T, K, 60, device=dev)
        tor, eor = workloads.top2_routing(T, E, 70)
        eor[eor == E - 1] = 0                     # the last expert stays empty, expert 0 gets two shares
        for mode in (dps.DPS_MODE_FAST, dps.DPS_MODE_FULL):
            y = dps.dps_moe_linear(mode, encs, x, torch.from_numpy(tor).to(dev), torch.from_numpy(eor).to(dev), p,
                                   r if mode else None)
            ref, rc = oracle.moe_linear(mode, encs, to_np_words(x), tor, eor, p_ref, r_ref, threads=8)
            assert rc == oracle.OK
            assert_close_to_oracle(y, ref, f"grouped E={E} N={N} mode={mode}")
            print(f"ok grouped E={E} N={N} K={K} T={T} mode={mode}")
    assert dps.dps_stream_status() == dps.DPS_OK
    print("all row-block cases passed")


@pytest.mark.gpu
@pytest.mark.parametrize("knobs", [
    {},
    {"DPS_FORCE_PATH": "pair", "DPS_PAIR_TOKENS": "192", "DPS_PAIR_SPLIT": "1"},
    {"DPS_FORCE_PATH": "pair", "DPS_PAIR_TOKENS": "256", "DPS_PAIR_SPLIT": "1"},
    {"DPS_FORCE_PATH": "pair", "DPS_PAIR_TOKENS": "256", "DPS_PAIR_SPLIT": "2"},
    {"DPS_FORCE_PATH": "umma", "DPS_FORCE_SPLIT": "1"},
    {"DPS_FORCE_PATH": "umma", "DPS_FORCE_SPLIT": "3"},
], ids=["default", "pair192", "pair256", "pair256_split2", "umma", "umma_split3"])
def test_ragged_shapes_in_child_process(knobs):
    env = dict(os.environ, DPS_DEBUG="1", PYTHONPATH=REPO, **knobs)
    out = subprocess.run([sys.executable, os.path.abspath(__file__)], cwd=REPO, env=env, capture_output=True,
                         text=True, timeout=600)
    assert out.returncode == 0, out.stdout[-2000:] + out.stderr[-4000:]
    assert "all row-block cases passed" in out.stdout
    assert out.stdout.count("ok dense") == 16 and out.stdout.count("ok grouped") == 4
    # what was asked for is what ran
    launches = [line for line in out.stderr.splitlines() if line.startswith("[dps]") and "grouped" not in line]
    assert len(launches) == 16
    path, tokens, split = (knobs.get(k) for k in ("DPS_FORCE_PATH", "DPS_PAIR_TOKENS", "DPS_PAIR_SPLIT"))
    if path:
        assert all(line.startswith(f"[dps] {path} ") for line in launches)
    if tokens:
        assert all(f"tokens={tokens} " in line for line in launches)
    split = split or knobs.get("DPS_FORCE_SPLIT")
    if split:       # (a K of fewer steps than the split needs keeps a smaller one)
        assert sum(f"split={split} " in line for line in launches) >= 12


if __name__ == "__main__":
    _cases()

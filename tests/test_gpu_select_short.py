"""The selection of short batches (one kernel) and of the next longer ones (four kernels) against a plain statement of
the rules: sizes around the warps and the keys per lane, ties on both sides, capacities from one to all candidates."""

import pytest
import torch

from paper_2406_00023_b200 import etr

pytestmark = pytest.mark.gpu


def expected(delta, mode, k, C):
    """[T, E] mask of the kept pairs: ties go to the lower expert, then to the lower token."""
    T, E = delta.shape
    cand = torch.ones(T, E, dtype=torch.bool)
    if mode == etr.MODE_TCR:
        order = torch.sort(delta, dim=1, descending=True, stable=True).indices
        cand = torch.zeros(T, E, dtype=torch.bool).scatter_(1, order[:, :k], True)
    kept = torch.zeros(T, E, dtype=torch.bool)
    for i in range(E):
        toks = cand[:, i].nonzero().flatten()
        best = torch.sort(delta[toks, i], descending=True, stable=True).indices[:C]
        kept[toks[best], i] = True
    return kept


@pytest.mark.parametrize("mode", [etr.MODE_TCR, etr.MODE_ECR])
@pytest.mark.parametrize("T,E,k,cap", [(1, 4, 1, 1), (31, 16, 2, 3), (33, 90, 1, 1), (128, 32, 2, 9), (129, 32, 3, 14),
                                       (256, 8, 2, 40), (257, 8, 2, 257), (511, 5, 2, 100), (512, 32, 2, 20),
                                       (513, 16, 2, 70), (64, 256, 1, 2), (64, 256, 3, 2)])
def test_selection(mode, T, E, k, cap):
    g = torch.Generator().manual_seed(T * E + k)
    cfg = etr.make_config(T=T, d=2048, D=8, E=E, k=k, h=64, capacity=cap, dtype=etr.BF16, mode=mode)
    b = etr.LayerBuffers(cfg)
    for ties in (False, True):
        delta = torch.randn(T, E, generator=g)
        if ties:
            delta = (delta * 2).round() / 2 + 0.0            # few values; + 0.0: no negative zeros, which order below zero
        b.block.fill_(0xFF)
        b.stats.zero_()
        etr.select(cfg, delta.cuda(), b.c.stats, b.route, b.c.ws)
        st, kept = b.read_stats(), expected(delta, mode, k, cap)
        Cs = etr.c_stride(cfg)
        rows = [[] for _ in range(T)]
        for i in range(E):
            toks = kept[:, i].nonzero().flatten().tolist()
            assert b.counts[i].item() == len(toks)
            assert b.slot_token.view(E, Cs)[i].tolist() == toks + [-1] * (Cs - len(toks))
            assert b.gate.view(E, Cs)[i].cpu().equal(torch.cat([delta[toks, i], torch.zeros(Cs - len(toks))]))
            for r, t in enumerate(toks):
                rows[t].append(i * Cs + r)
        flat = [r for t in rows for r in t]
        assert b.tok_ptr.tolist() == [0] + torch.tensor([len(t) for t in rows]).cumsum(0).tolist()
        assert b.tok_row[:len(flat)].tolist() == flat
        want = torch.sort(delta, dim=1, descending=True, stable=True).indices[:, :k] if mode == etr.MODE_TCR else torch.full((T, k), -1)
        assert b.topk_idx.cpu().long().equal(want)
        cands = T * k if mode == etr.MODE_TCR else T * E
        assert (st.rows_total, st.dropped, st.unrouted, st.C) == (len(flat), cands - len(flat), sum(not t for t in rows), cap)

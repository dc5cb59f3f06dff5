"""GPU: rows reset between calls carry the empty prefix's mask into every call that follows,
and the other rows keep theirs (the mask ids stay current across a reset)."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import Oracle, Vocab
from workloads import grammars

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def psc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_03065_gb300 import build, psc as mod
    build.build()
    mod.load()
    return mod


@pytest.mark.parametrize("global_tables", [False, True])
@pytest.mark.parametrize("call", ["fill_mask", "fill_apply", "argmax", "choose", "step", "advance"])
@pytest.mark.parametrize("rows", [[0], [5], [1, 3], None, [2, -1, 99]])
def test_masks_after_reset(psc, rows, call, global_tables):
    g = grammars.json_grammar().text()
    toks = [bytes([c]) for c in b'[]{}:,"0123456789truefalsn -.e'] + [b'[1', b'{"', b'"]', b""]
    V, B = len(toks), 6
    h = psc.psc_compile(g, toks, V - 1, global_tables=global_tables)
    o, voc = Oracle(g), Vocab.from_list(toks, V - 1)
    st = psc.psc_state_init(h, B, 16)
    first = [toks.index(t) for t in (b"[", b"{", b'"', b"1", b"[1", b'{"')]
    psc.psc_advance(h, st, torch.tensor(first, dtype=torch.int32, device="cuda"))
    ocs = []
    for b, t in enumerate(first):
        oc = o.initial()
        if not (rows is None or b in rows):
            o.advance_tokens(oc, voc, [t])
        ocs.append(oc)
    psc.psc_state_reset(st, None if rows is None else torch.tensor(rows, dtype=torch.int32, device="cuda"))
    ref = o.masks(ocs, voc)
    bits = np.unpackbits(ref.view(np.uint8), axis=-1, bitorder="little")[:, :V].astype(bool)
    x = torch.randn(B, V, generator=torch.Generator().manual_seed(3)).cuda()
    want = np.where(bits, x.cpu().numpy(), -np.inf)
    bm = torch.zeros(B, h.W, dtype=torch.int32, device="cuda")
    tok = torch.zeros(B, dtype=torch.int32, device="cuda")
    status = torch.zeros(B, dtype=torch.int32, device="cuda")
    if call == "fill_mask":
        psc.psc_fill_mask(h, st, bm)
    elif call == "fill_apply":
        psc.psc_fill_apply(h, st, x, bm)
    elif call == "argmax":
        psc.psc_argmax_masked(h, st, x, tok)
    elif call == "choose":
        psc.psc_fill_apply_argmax(h, st, x, tok, bm)
    elif call == "step":
        psc.psc_decode_step(h, st, x, tok, bm)
    else:   # the advance checks its tokens against the rows' masks
        psc.psc_advance(h, st, torch.full((B,), toks.index(b"]"), dtype=torch.int32, device="cuda"), status)
        np.testing.assert_array_equal(status.cpu().numpy() == psc.ROW_OK, bits[:, toks.index(b"]")])
    if call in ("fill_mask", "fill_apply", "choose", "step"):
        np.testing.assert_array_equal(bm.cpu().numpy().view(np.uint32), ref)
    if call in ("fill_apply", "choose", "step"):
        np.testing.assert_array_equal(x.cpu().numpy(), want)
    if call in ("argmax", "choose", "step"):
        np.testing.assert_array_equal(tok.cpu().numpy(), np.argmax(want, axis=1))

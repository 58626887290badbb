"""Signature rows of tokens that repeat one another to the grammar, against the plain Python oracle: narrow, wide and odd row widths,
short rows behind long ones, rows that do not fit (no GPU needed)."""
import numpy as np
import pytest

import synth
from oracle import offline
from test_offline_host import library_signatures


@pytest.mark.parametrize("row_words", [4, 9, 64, 67, 300])
def test_rows_of_tokens_that_read_alike(row_words):
    spec = synth.grammars.arithmetic_grammar()
    base = synth.grammars.toy_vocabulary(spec, max_len=2, extra=40)
    order = np.random.RandomState(row_words).randint(0, len(base), 700)
    tokens = [base[i] for i in order]
    _, sig, words, rc = library_signatures(spec, tokens, row_words)
    names, start, prods = spec
    _, _, want = offline.token_classes(offline.Grammar(len(names), start, prods), tokens)
    assert np.array_equal(words, [len(w) for w in want])
    for row, w in zip(sig, want):
        full = [len(w)] + list(w) if len(w) + 1 <= row_words else []
        assert row.tolist() == full + [0] * (row_words - len(full))
    assert rc == (0 if max(len(w) for w in want) + 1 <= row_words else -2)

"""How many query tiles a CTA of the tree attention takes (host rule): one
where pairs were measured slower (one tile per kv head; a wave of pairs and a
tail against two waves of single tiles; half-empty pairs over a long context),
two where they were measured faster."""
import pytest

from paper_2608_13524_gb300 import dart

SMS = 152
# (nseq, B, C) with 32 query and 8 kv heads (32 rows per tile); µs measured on GB300: pairs, single tiles
ONE = [(24, 32, 2048), (45, 32, 300), (64, 32, 2048), (11, 96, 300), (11, 96, 2048), (7, 160, 2048), (5, 224, 8192),
       (25, 96, 2048), (38, 96, 8192), (13, 160, 8192), (4, 64, 2048), (1, 64, 2048)]
TWO = [(16, 64, 2048), (45, 64, 300), (7, 96, 2048), (13, 96, 8192), (28, 96, 0), (8, 512, 2048), (8, 512, 16384),
       (11, 128, 2048), (9, 160, 300), (45, 352, 2048), (8, 1024, 0)]


@pytest.mark.parametrize("shape,want", [(s, 1) for s in ONE] + [(s, 2) for s in TWO])
def test_tiles_per_cta(shape, want):
    nseq, B, C = shape
    cfg = dart.make_attn_config(nseq, B, C, 32, 8, 128, 1e6, 0.1)
    assert dart.dart_tree_attention_tiles(cfg, SMS) == want


def test_tiles_of_other_groupings():
    # 128 rows per tile without grouped heads: 192 tiles, one per head
    assert dart.dart_tree_attention_tiles(dart.make_attn_config(8, 128, 1024, 24, 24, 128, 1e6, 0.1), SMS) == 1
    # 8 rows per tile with 16 heads per kv head
    assert dart.dart_tree_attention_tiles(dart.make_attn_config(80, 8, 1024, 32, 2, 128, 1e6, 0.1), SMS) == 1
    assert dart.dart_tree_attention_tiles(dart.make_attn_config(80, 16, 1024, 32, 2, 128, 1e6, 0.1), SMS) == 2
    assert dart.dart_tree_attention_tiles(dart.make_attn_config(8, 0, 0, 32, 8, 128, 1e6, 0.1), SMS) == 0

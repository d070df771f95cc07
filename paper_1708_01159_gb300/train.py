"""Training the per-level decision tree (Section 4.1, Section 4.2).

  collect  -- on a GPU: run the per-level timing harness (bfs_profile_levels)
              over a set of generated graphs and roots and write one CSV row
              per (graph, root, level): the 26 integer features and the median
              time of every variant expanding that level from the same state.
  train    -- label every level with its fastest variant, fit a CART tree
              (Gini impurity, scikit-learn) and export it in the integer text
              format bfs_load_tree reads: thresholds become floor(t) (the
              features are integers, so x <= t and x <= floor(t) agree), and a
              leaf whose two largest class weights tie is marked unknown (-1),
              the case Section 4.1 resolves by repeating the previous level's
              choice.
  evaluate -- per traversal, the time of the tree's schedule (unknown rule
              applied), of the best fixed variant and of every variant, each
              relative to the per-level optimum (the shape of Table 2).
  cv       -- k-fold cross-validation by graph over feature sets, weightings
              and depths.
  holdout  -- each generator family (R-MAT, directed R-MAT, grid, ER and the
              other shapes) held out in turn: trained on the others, evaluated on it (Section 4.4).
  level-split -- the paper's random 70/30 split over levels: held-out
              per-level accuracy, for comparison with its reported accuracy.

The benchmark's own graph (R-MAT scale 22, seed 1001) is never in the
training set. Graphs are split into train and test sets by graph, since the
levels of one traversal are correlated.

  python -m paper_1708_01159_gb300.train collect --out levels.csv
  python -m paper_1708_01159_gb300.train train --csv levels.csv --out trees/default.tree
  python -m paper_1708_01159_gb300.train evaluate --csv levels.csv --tree trees/default.tree
  python -m paper_1708_01159_gb300.train level-split --csv levels.csv
  python -m paper_1708_01159_gb300.train holdout --csv levels.csv
"""
from __future__ import annotations

import argparse
import csv
import math
import os
import sys
import time

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, os.path.dirname(HERE))

from paper_1708_01159_gb300 import FEATURES, NUM_FEATURES, NUM_VARIANTS, VARIANTS  # noqa: E402

LEVEL0_DEFAULT = 3  # Section 4.1: unknown at the first level -> edge list (edge-centric push)

# Feature sets (indices into FEATURES):
#   paper -- Section 4.2's best model: graph size, % of vertices discovered,
#            out-degree distribution, vertices in the frontier
#   m1    -- every feature Section 4.1 lists (frontier and discovered both
#            absolute and as a share of the vertices)
#   ext   -- m1 plus the frontier's edge count and the level index
#   *_io  -- the same plus the in-degree and total-degree summaries (Section
#            4.1 names the distribution of in-, out- or total degree), which
#            tell directed graphs apart
FEATURE_SETS = {
    "paper": [0, 1, 2, 3, 4, 5, 6, 7, 8, 11],
    "paper_io": [0, 1, 2, 3, 4, 5, 6, 7, 8, 11] + list(range(14, 26)),
    "m1": list(range(12)),
    "ext": list(range(14)),
    "ext_io": list(range(26)),
}

# Training graphs: (name, generator kwargs). Seeds start at 3000; the
# benchmark graph uses seed 1001 and is excluded by construction.
TRAIN_GRAPHS = [
    ("rmat", dict(scale=16, edge_factor=16, seed=3001)),
    ("rmat", dict(scale=18, edge_factor=8, seed=3002)),
    ("rmat", dict(scale=18, edge_factor=32, seed=3003)),
    ("rmat", dict(scale=20, edge_factor=16, seed=3004)),
    ("rmat", dict(scale=20, edge_factor=4, seed=3005)),
    ("rmat", dict(scale=21, edge_factor=16, seed=3006, permute=True)),
    ("rmat", dict(scale=22, edge_factor=16, seed=3007)),
    ("rmat", dict(scale=22, edge_factor=8, seed=3008)),
    ("rmat", dict(scale=19, edge_factor=16, seed=3009, a=0.45, b=0.15, c=0.15)),
    ("rmat", dict(scale=21, edge_factor=24, seed=3010, a=0.50, b=0.20, c=0.20)),
    ("grid", dict(rows=512, cols=512, drop=0.1, seed=3011)),
    ("grid", dict(rows=1024, cols=1024, drop=0.1, seed=3012)),
    ("grid", dict(rows=2048, cols=2048, drop=0.2, seed=3013)),
    ("grid", dict(rows=1500, cols=3000, drop=0.05, seed=3014)),
    ("er", dict(n=1 << 20, avg_degree=4.0, seed=3015)),
    ("er", dict(n=1 << 21, avg_degree=8.0, seed=3016)),
    ("er", dict(n=1 << 22, avg_degree=16.0, seed=3017)),
    ("er", dict(n=1 << 18, avg_degree=32.0, seed=3018)),
    # the workloads' own sizes, other seeds: 16.8M-vertex grids, 2^23 ER, scale 23 R-MAT
    ("grid", dict(rows=4096, cols=4096, drop=0.1, seed=3019)),
    ("grid", dict(rows=3000, cols=3000, drop=0.15, seed=3020)),
    ("er", dict(n=1 << 23, avg_degree=8.0, seed=3021)),
    ("rmat", dict(scale=23, edge_factor=16, seed=3022)),
    ("rmat", dict(scale=17, edge_factor=16, seed=3023, permute=True)),
    # directed R-MAT (not symmetrised): with b != c the in- and out-degree
    # distributions differ, and pull scans the transpose
    ("rmat", dict(scale=18, edge_factor=16, seed=3024, directed=True, b=0.30, c=0.08)),
    ("rmat", dict(scale=20, edge_factor=8, seed=3025, directed=True, b=0.08, c=0.30)),
    ("rmat", dict(scale=21, edge_factor=16, seed=3026, directed=True)),
    ("rmat", dict(scale=22, edge_factor=8, seed=3027, directed=True, b=0.25, c=0.13)),
    # small graphs, where the launch-bound levels and the few wide ones trade places
    ("rmat", dict(scale=12, edge_factor=16, seed=3028)),
    ("rmat", dict(scale=13, edge_factor=8, seed=3029)),
    ("rmat", dict(scale=14, edge_factor=16, seed=3030)),
    ("rmat", dict(scale=14, edge_factor=32, seed=3031, permute=True)),
    ("rmat", dict(scale=15, edge_factor=24, seed=3032)),
    ("rmat", dict(scale=13, edge_factor=16, seed=3033, directed=True, b=0.25, c=0.13)),
    ("rmat", dict(scale=17, edge_factor=16, seed=3034, directed=True)),
    ("rmat", dict(scale=19, edge_factor=16, seed=3035, directed=True)),
    ("rmat", dict(scale=20, edge_factor=16, seed=3036, directed=True)),
    ("er", dict(n=6000, avg_degree=16.0, seed=3037)),
    ("er", dict(n=1 << 14, avg_degree=8.0, seed=3038)),
    ("er", dict(n=1 << 16, avg_degree=24.0, seed=3039)),
    ("er", dict(n=200000, avg_degree=4.0, seed=3040)),
    ("er", dict(n=700000, avg_degree=16.0, seed=3041)),
    ("grid", dict(rows=64, cols=200, drop=0.1, seed=3042)),
    ("er", dict(n=4096, avg_degree=4.0, seed=3043)),
    ("er", dict(n=8192, avg_degree=8.0, seed=3044)),
    ("er", dict(n=10000, avg_degree=32.0, seed=3045)),
    ("er", dict(n=30000, avg_degree=16.0, seed=3046)),
    ("er", dict(n=50000, avg_degree=8.0, seed=3047)),
    ("er", dict(n=120000, avg_degree=24.0, seed=3048)),
    ("er", dict(n=400000, avg_degree=8.0, seed=3049)),
    ("er", dict(n=1500000, avg_degree=4.0, seed=3050)),
    ("rmat", dict(scale=12, edge_factor=32, seed=3051)),
    ("rmat", dict(scale=13, edge_factor=24, seed=3052, permute=True)),
    ("rmat", dict(scale=15, edge_factor=8, seed=3053)),
    ("rmat", dict(scale=16, edge_factor=32, seed=3054)),
    ("rmat", dict(scale=14, edge_factor=8, seed=3055, directed=True)),
    ("rmat", dict(scale=16, edge_factor=8, seed=3056, directed=True)),
    ("rmat", dict(scale=18, edge_factor=24, seed=3057, directed=True)),
    ("rmat", dict(scale=21, edge_factor=8, seed=3058)),
    ("grid", dict(rows=40, cols=37, drop=0.1, seed=3059)),
    ("er", dict(n=2097152, avg_degree=16.0, seed=3060)),
    ("er", dict(n=1048576, avg_degree=16.0, seed=3061)),
    ("er", dict(n=1048576, avg_degree=32.0, seed=3062)),
    ("er", dict(n=524288, avg_degree=16.0, seed=3063)),
    ("er", dict(n=262144, avg_degree=8.0, seed=3064)),
    ("er", dict(n=262144, avg_degree=16.0, seed=3065)),
    ("er", dict(n=3000000, avg_degree=8.0, seed=3066)),
    ("er", dict(n=4194304, avg_degree=4.0, seed=3067)),
    ("er", dict(n=4194304, avg_degree=8.0, seed=3068)),
    ("er", dict(n=131072, avg_degree=16.0, seed=3069)),
    ("er", dict(n=65536, avg_degree=8.0, seed=3070)),
    ("er", dict(n=32768, avg_degree=16.0, seed=3071)),
    ("er", dict(n=8192, avg_degree=24.0, seed=3072)),
    ("er", dict(n=900000, avg_degree=4.0, seed=3073)),
    ("er", dict(n=1048576, avg_degree=24.0, seed=3074)),
    ("rmat", dict(scale=20, edge_factor=16, seed=3075)),
    ("rmat", dict(scale=18, edge_factor=16, seed=3076)),
    ("rmat", dict(scale=17, edge_factor=8, seed=3077)),
    ("rmat", dict(scale=16, edge_factor=16, seed=3078, permute=True)),
    ("rmat", dict(scale=19, edge_factor=24, seed=3079)),
    ("rmat", dict(scale=21, edge_factor=16, seed=3080)),
    ("rmat", dict(scale=12, edge_factor=8, seed=3081)),
    ("rmat", dict(scale=20, edge_factor=8, seed=3082, directed=True)),
    ("rmat", dict(scale=18, edge_factor=8, seed=3083, directed=True)),
    ("rmat", dict(scale=15, edge_factor=16, seed=3084, directed=True)),
    ("rmat", dict(scale=12, edge_factor=16, seed=3085, directed=True)),
    ("rmat", dict(scale=20, edge_factor=24, seed=3086, directed=True)),
    ("rmat", dict(scale=16, edge_factor=4, seed=3087)),
    ("rmat", dict(scale=11, edge_factor=8, seed=3088)),
    ("rmat", dict(scale=11, edge_factor=8, seed=3089, permute=True)),
    ("rmat", dict(scale=11, edge_factor=16, seed=3090)),
    ("rmat", dict(scale=11, edge_factor=16, seed=3091, permute=True)),
    ("rmat", dict(scale=12, edge_factor=4, seed=3092)),
    ("rmat", dict(scale=12, edge_factor=4, seed=3093, permute=True)),
    ("rmat", dict(scale=12, edge_factor=4, seed=3094)),
    ("rmat", dict(scale=12, edge_factor=4, seed=3095, permute=True)),
    ("rmat", dict(scale=12, edge_factor=8, seed=3096)),
    ("rmat", dict(scale=12, edge_factor=8, seed=3097, permute=True)),
    ("rmat", dict(scale=12, edge_factor=16, seed=3098)),
    ("rmat", dict(scale=12, edge_factor=16, seed=3099, permute=True)),
    ("rmat", dict(scale=13, edge_factor=4, seed=3100)),
    ("rmat", dict(scale=13, edge_factor=4, seed=3101, permute=True)),
    ("rmat", dict(scale=13, edge_factor=4, seed=3102)),
    ("rmat", dict(scale=13, edge_factor=4, seed=3103, permute=True)),
    ("rmat", dict(scale=13, edge_factor=8, seed=3104)),
    ("rmat", dict(scale=13, edge_factor=8, seed=3105, permute=True)),
    ("rmat", dict(scale=13, edge_factor=16, seed=3106)),
    ("rmat", dict(scale=13, edge_factor=16, seed=3107, permute=True)),
    ("rmat", dict(scale=14, edge_factor=4, seed=3108)),
    ("rmat", dict(scale=14, edge_factor=4, seed=3109, permute=True)),
    ("rmat", dict(scale=14, edge_factor=8, seed=3110)),
    ("rmat", dict(scale=14, edge_factor=8, seed=3111, permute=True)),
    ("rmat", dict(scale=12, edge_factor=24, seed=3112)),
    ("rmat", dict(scale=12, edge_factor=24, seed=3113, permute=True)),
    ("rmat", dict(scale=11, edge_factor=32, seed=3114)),
    ("rmat", dict(scale=11, edge_factor=32, seed=3115, permute=True)),
    # other shapes: a tree trained on R-MAT, grids and Erdos-Renyi alone pulled on
    # stars (114 times the time of its predecessor's push) and on chains of cliques
    ("smallworld", dict(n=4096, k=8, beta=0.1, seed=3116)),
    ("smallworld", dict(n=16384, k=6, beta=0.01, seed=3117)),
    ("smallworld", dict(n=30000, k=10, beta=0.1, seed=3118)),
    ("smallworld", dict(n=131072, k=5, beta=0.05, seed=3119)),
    ("smallworld", dict(n=524288, k=8, beta=0.2, seed=3120)),
    ("smallworld", dict(n=1000000, k=6, beta=0.3, seed=3121)),
    ("smallworld", dict(n=2097152, k=5, beta=0.02, seed=3122)),
    ("growing", dict(n=8192, k=4, seed=3123)),
    ("growing", dict(n=32768, k=8, seed=3124)),
    ("growing", dict(n=262144, k=6, seed=3125)),
    ("growing", dict(n=1048576, k=8, seed=3126)),
    ("growing", dict(n=2097152, k=5, seed=3127)),
    ("powerlaw", dict(n=8192, degree=8, exponent=2.3, seed=3128)),
    ("powerlaw", dict(n=65536, degree=12, exponent=2.4, seed=3129)),
    ("powerlaw", dict(n=262144, degree=8, exponent=2.2, seed=3130)),
    ("powerlaw", dict(n=524288, degree=24, exponent=2.6, seed=3131)),
    ("powerlaw", dict(n=1048576, degree=16, exponent=2.8, seed=3132)),
    ("powerlaw", dict(n=2097152, degree=8, exponent=2.1, seed=3133)),
    ("powerlaw", dict(n=32768, degree=8, exponent=2.3, seed=3134, directed=True)),
    ("powerlaw", dict(n=262144, degree=16, exponent=2.4, seed=3135, directed=True)),
    ("powerlaw", dict(n=1048576, degree=8, exponent=2.2, seed=3136, directed=True)),
    ("moves", dict(dims=(200, 200), radius=1, seed=3137)),
    ("moves", dict(dims=(400, 400), radius=2, seed=3138)),
    ("moves", dict(dims=(700, 700), radius=2, seed=3139)),
    ("moves", dict(dims=(250, 250), radius=3, seed=3140)),
    ("moves", dict(dims=(128, 128), radius=4, seed=3141)),
    ("moves", dict(dims=(1500, 200), radius=2, seed=3142)),
    ("moves", dict(dims=(30, 30, 30), radius=1, seed=3143)),
    ("moves", dict(dims=(90, 90, 90), radius=1, seed=3144)),
    ("moves", dict(dims=(200, 60, 60), radius=1, seed=3145)),
    ("moves", dict(dims=(50000,), radius=100, seed=3146)),
    ("cliques", dict(count=300, size=16, seed=3147)),
    ("cliques", dict(count=300, size=64, seed=3148)),
    ("cliques", dict(count=100, size=200, seed=3149)),
    ("cliques", dict(count=300, size=10, seed=3150)),
    ("cliques", dict(count=60, size=400, seed=3151)),
    ("cliques", dict(count=20, size=1000, seed=3152)),
    ("stars", dict(n=3000, hubs=1, seed=3153)),
    ("stars", dict(n=200000, hubs=1, seed=3154)),
    ("stars", dict(n=500000, hubs=20, seed=3155)),
    ("stars", dict(n=2000000, hubs=1000, seed=3156)),
    ("stars", dict(n=100000, hubs=300, seed=3157)),
    ("stars", dict(n=50000, hubs=3, seed=3158)),
    ("stars", dict(n=20000, hubs=10, links=2, seed=3159)),
    ("stars", dict(n=400000, hubs=50, links=2, seed=3160)),
    ("stars", dict(n=1000000, hubs=2000, links=2, seed=3161)),
    ("layers", dict(count=30, width=5000, k=8, seed=3162, directed=True)),
    ("layers", dict(count=200, width=3000, k=12, seed=3163, directed=True)),
    ("layers", dict(count=8, width=100000, k=16, seed=3164, directed=True)),
    ("layers", dict(count=100, width=400, k=10, seed=3165, directed=True)),
    ("layers", dict(count=20, width=100000, k=9, seed=3166, directed=True)),
    ("layers", dict(count=300, width=20000, k=10, seed=3167)),
    ("layers", dict(count=60, width=1000, k=20, seed=3168)),
    ("bipartite", dict(left=300, right=3000, edges=50000, seed=3169)),
    ("bipartite", dict(left=500, right=200000, edges=2000000, seed=3170)),
    ("bipartite", dict(left=50000, right=50000, edges=1000000, seed=3171)),
    ("bipartite", dict(left=5000, right=500000, edges=4000000, seed=3172)),
    ("bipartite", dict(left=20, right=100000, edges=300000, seed=3173)),
    ("regular", dict(n=65536, k=12, seed=3174)),
    ("regular", dict(n=262144, k=10, seed=3175)),
    ("regular", dict(n=1048576, k=16, seed=3176)),
    ("regular", dict(n=3000, k=200, seed=3177)),
    ("regular", dict(n=20000, k=64, seed=3178)),
    ("rmat", dict(scale=14, edge_factor=16, a=0.45, b=0.22, c=0.22, seed=3179)),
    ("rmat", dict(scale=17, edge_factor=8, a=0.45, b=0.22, c=0.22, seed=3180)),
    ("rmat", dict(scale=21, edge_factor=12, a=0.45, b=0.22, c=0.22, seed=3181)),
    ("rmat", dict(scale=16, edge_factor=16, a=0.7, b=0.1, c=0.1, seed=3182)),
    ("rmat", dict(scale=19, edge_factor=16, a=0.7, b=0.1, c=0.1, seed=3183)),
    ("rmat", dict(scale=20, edge_factor=2, seed=3184)),
    ("rmat", dict(scale=22, edge_factor=4, seed=3185)),
    ("rmat", dict(scale=17, edge_factor=8, a=0.45, b=0.22, c=0.22, seed=3186, directed=True)),
    ("er", dict(n=262144, avg_degree=1.5, seed=3187)),
    ("er", dict(n=2000, avg_degree=100.0, seed=3188)),
    ("stars", dict(n=10000, hubs=2, seed=3189)),
    ("stars", dict(n=30000, hubs=30, seed=3190)),
    ("stars", dict(n=150000, hubs=5, seed=3191)),
    ("stars", dict(n=300000, hubs=100, seed=3192)),
    ("stars", dict(n=1500000, hubs=150, seed=3193)),
    ("stars", dict(n=4000, hubs=4, links=2, seed=3194)),
    ("stars", dict(n=60000, hubs=6, links=3, seed=3195)),
    ("stars", dict(n=100000, hubs=40, links=2, seed=3196)),
    ("stars", dict(n=200000, hubs=10, links=4, seed=3197)),
    ("stars", dict(n=800000, hubs=20, links=2, seed=3198)),
    ("stars", dict(n=1200000, hubs=200, links=3, seed=3199)),
    ("tree", dict(n=100000, arity=10, seed=3200)),
    ("tree", dict(n=1000000, arity=30, seed=3201)),
    ("tree", dict(n=500000, arity=100, seed=3202)),
    ("tree", dict(n=200000, arity=1000, seed=3203)),
    ("tree", dict(n=1000000, arity=500, seed=3204)),
    ("tree", dict(n=30000, arity=50, seed=3205)),
    ("growing", dict(n=100000, k=1, seed=3206)),
    ("growing", dict(n=1500000, k=1, seed=3207)),
    ("growing", dict(n=400000, k=2, seed=3208)),
    ("growing", dict(n=3000000, k=3, seed=3209)),
    ("growing", dict(n=500000, k=16, seed=3210)),
    ("hubs", dict(n=20000, degree=4, hubs=2, share=0.5, seed=3211)),
    ("hubs", dict(n=100000, degree=3, hubs=10, share=0.2, seed=3212)),
    ("hubs", dict(n=400000, degree=8, hubs=5, share=0.05, seed=3213)),
    ("hubs", dict(n=1000000, degree=2, hubs=50, share=0.02, seed=3214)),
    ("hubs", dict(n=1000000, degree=6, hubs=1, share=0.9, seed=3215)),
    ("hubs", dict(n=200000, degree=1, hubs=30, share=0.03, seed=3216)),
    ("components", dict(count=500, size=100, degree=10, seed=3217)),
    ("components", dict(count=20, size=10000, degree=12, seed=3218)),
    ("components", dict(count=4, size=300000, degree=10, seed=3219)),
    ("components", dict(count=3000, size=400, degree=20, seed=3220)),
    ("cliques", dict(count=150, size=100, seed=3221)),
    ("cliques", dict(count=8, size=2000, seed=3222)),
    ("cliques", dict(count=400, size=30, seed=3223)),
    ("bipartite", dict(left=100, right=1000000, edges=3000000, seed=3224)),
    ("bipartite", dict(left=2000, right=100000, edges=500000, seed=3225)),
    ("bipartite", dict(left=1000000, right=1000000, edges=8000000, seed=3226)),
    ("layers", dict(count=12, width=300000, k=12, seed=3227)),
    ("layers", dict(count=150, width=8000, k=9, seed=3228)),
    ("rmat", dict(scale=21, edge_factor=3, seed=3229)),
    ("rmat", dict(scale=23, edge_factor=8, seed=3230)),
    ("rmat", dict(scale=18, edge_factor=2, seed=3231)),
    # R-MAT on vertex counts that are no power of two
    ("rmatcut", dict(n=5000, edge_factor=8, seed=3232)),
    ("rmatcut", dict(n=5657, edge_factor=24, seed=3233)),
    ("rmatcut", dict(n=9187, edge_factor=12, seed=3234)),
    ("rmatcut", dict(n=10438, edge_factor=16, seed=3235, directed=True)),
    ("rmatcut", dict(n=17221, edge_factor=4, seed=3236)),
    ("rmatcut", dict(n=17221, edge_factor=8, seed=3237)),
    ("rmatcut", dict(n=24000, edge_factor=16, seed=3238)),
    ("rmatcut", dict(n=24000, edge_factor=6, seed=3239, directed=True)),
    ("rmatcut", dict(n=45098, edge_factor=8, seed=3240, directed=True)),
    ("rmatcut", dict(n=45098, edge_factor=24, seed=3241)),
    ("rmatcut", dict(n=70000, edge_factor=4, seed=3242)),
    ("rmatcut", dict(n=90000, edge_factor=12, seed=3243)),
    ("rmatcut", dict(n=100003, edge_factor=6, seed=3244, directed=True)),
    ("rmatcut", dict(n=182362, edge_factor=16, seed=3245, directed=True)),
    ("rmatcut", dict(n=182362, edge_factor=4, seed=3246)),
    ("rmatcut", dict(n=300000, edge_factor=8, seed=3247)),
    ("rmatcut", dict(n=300000, edge_factor=3, seed=3248)),
    ("rmatcut", dict(n=419000, edge_factor=16, seed=3249)),
    ("rmatcut", dict(n=419000, edge_factor=8, seed=3250, directed=True)),
    ("rmatcut", dict(n=700000, edge_factor=4, seed=3251)),
    ("rmatcut", dict(n=700000, edge_factor=12, seed=3252, directed=True)),
    ("rmatcut", dict(n=1000003, edge_factor=8, seed=3253, directed=True)),
    ("rmatcut", dict(n=1100000, edge_factor=12, seed=3254)),
    ("rmatcut", dict(n=1234844, edge_factor=3, seed=3255)),
    ("rmatcut", dict(n=1472023, edge_factor=16, seed=3256)),
    ("rmatcut", dict(n=1472023, edge_factor=6, seed=3257, directed=True)),
    ("rmatcut", dict(n=2500000, edge_factor=4, seed=3258)),
    ("rmatcut", dict(n=2500000, edge_factor=8, seed=3259, directed=True)),
    ("rmatcut", dict(n=3000000, edge_factor=12, seed=3260)),
    ("rmatcut", dict(n=3500000, edge_factor=2, seed=3261)),
    ("rmatcut", dict(n=3500000, edge_factor=16, seed=3262)),
    ("er", dict(n=9742, avg_degree=4.0, seed=3263)),
    ("er", dict(n=16384, avg_degree=4.0, seed=3264)),
    ("er", dict(n=32768, avg_degree=4.0, seed=3265)),
    ("er", dict(n=76173, avg_degree=4.0, seed=3266)),
    ("er", dict(n=382885, avg_degree=4.0, seed=3267)),
    ("er", dict(n=3000000, avg_degree=16.0, seed=3268)),
    ("er", dict(n=2300000, avg_degree=12.0, seed=3269)),
    ("er", dict(n=600000, avg_degree=6.0, seed=3270)),
    ("rmatn", dict(n=86849, degree=8, seed=3277, directed=True)),
    ("rmatn", dict(n=23858, degree=4, seed=3278, directed=True)),
    ("rmatn", dict(n=1244092, degree=4, seed=3279)),
    ("rmatn", dict(n=38157, degree=8, seed=3280)),
    ("rmatn", dict(n=1533801, degree=4, seed=3281)),
    ("rmatn", dict(n=37090, degree=16, seed=3282, directed=True)),
    ("rmatn", dict(n=414929, degree=24, seed=3283, directed=True)),
    ("rmatn", dict(n=49906, degree=24, seed=3284)),
    ("rmatn", dict(n=2103978, degree=8, seed=3285)),
    ("rmatn", dict(n=11549, degree=4, seed=3286)),
    ("rmatn", dict(n=5746, degree=4, seed=3287, directed=True)),
    ("rmatn", dict(n=115531, degree=16, seed=3288, directed=True)),
    ("rmatn", dict(n=6219, degree=24, seed=3289)),
    ("rmatn", dict(n=51459, degree=24, seed=3290)),
    ("rmatn", dict(n=1426130, degree=8, seed=3291)),
    ("rmatn", dict(n=15831, degree=4, seed=3292, directed=True)),
    ("rmatn", dict(n=491287, degree=8, seed=3293, directed=True)),
    ("rmatn", dict(n=1448048, degree=8, seed=3294)),
    ("rmatn", dict(n=1672029, degree=8, seed=3295)),
    ("rmatn", dict(n=26174, degree=32, seed=3296)),
    ("rmatn", dict(n=5446, degree=24, seed=3297, directed=True)),
    ("rmatn", dict(n=1418024, degree=8, seed=3298, directed=True)),
    ("rmatn", dict(n=5879, degree=8, seed=3299)),
    ("rmatn", dict(n=1084909, degree=4, seed=3300)),
    ("rmatn", dict(n=4782, degree=8, seed=3301)),
    ("rmatn", dict(n=526615, degree=32, seed=3302, directed=True)),
    ("rmatn", dict(n=8577, degree=16, seed=3303, directed=True)),
    ("rmatn", dict(n=4202, degree=32, seed=3304)),
    ("rmatn", dict(n=186293, degree=32, seed=3305)),
    ("rmatn", dict(n=15633, degree=4, seed=3306)),
    ("rmatn", dict(n=1476007, degree=4, seed=3307, directed=True)),
    ("rmatn", dict(n=144102, degree=4, seed=3308, directed=True)),
    ("rmatn", dict(n=111440, degree=16, seed=3309)),
    ("rmatn", dict(n=108494, degree=4, seed=3310)),
    ("rmatn", dict(n=65443, degree=8, seed=3311)),
    ("rmatn", dict(n=14550, degree=32, seed=3312, directed=True)),
    ("rmatn", dict(n=7585, degree=16, seed=3313, directed=True)),
    ("rmatn", dict(n=10684, degree=16, seed=3314)),
    ("rmatn", dict(n=472001, degree=4, seed=3315)),
    ("rmatn", dict(n=5855, degree=16, seed=3316)),
    ("rmatn", dict(n=371224, degree=32, seed=3317, directed=True)),
    ("rmatn", dict(n=10966, degree=8, seed=3318, directed=True)),
    ("rmatn", dict(n=528873, degree=16, seed=3319)),
    ("rmatn", dict(n=2959984, degree=4, seed=3320)),
    ("rmatn", dict(n=1261431, degree=8, seed=3321)),
    ("rmatn", dict(n=2170334, degree=4, seed=3322, directed=True)),
    ("rmatn", dict(n=11904, degree=16, seed=3323, directed=True)),
    ("rmatn", dict(n=5440, degree=8, seed=3324)),
    ("rmatn", dict(n=1083903, degree=16, seed=3325)),
    ("rmatn", dict(n=201053, degree=32, seed=3326)),
    ("rmatn", dict(n=382380, degree=32, seed=3327, directed=True)),
    ("rmatn", dict(n=40457, degree=32, seed=3328, directed=True)),
    ("rmatn", dict(n=1374815, degree=8, seed=3329)),
    ("rmatn", dict(n=80394, degree=8, seed=3330)),
    ("rmatn", dict(n=15198, degree=16, seed=3331)),
    ("rmatn", dict(n=560544, degree=8, seed=3332, directed=True)),
    ("rmatn", dict(n=798663, degree=8, seed=3333, directed=True)),
    ("rmatn", dict(n=4112, degree=4, seed=3334)),
    ("rmatn", dict(n=16740, degree=8, seed=3335)),
    ("rmatn", dict(n=24255, degree=32, seed=3336)),
    ("rmatn", dict(n=7358, degree=24, seed=3337, directed=True)),
    ("rmatn", dict(n=26822, degree=16, seed=3338, directed=True)),
    ("rmatn", dict(n=722130, degree=4, seed=3339)),
    ("rmatn", dict(n=50690, degree=16, seed=3340)),
    ("rmatn", dict(n=842941, degree=8, seed=3341)),
    ("rmatn", dict(n=40159, degree=32, seed=3342, directed=True)),
    ("rmatn", dict(n=21065, degree=24, seed=3343, directed=True)),
    ("rmatn", dict(n=6342, degree=24, seed=3344)),
    ("rmatn", dict(n=18792, degree=32, seed=3345)),
    ("rmatn", dict(n=57657, degree=8, seed=3346)),
    ("rmatn", dict(n=2241902, degree=16, seed=3347, directed=True)),
    ("rmatn", dict(n=46826, degree=24, seed=3348, directed=True)),
    ("er", dict(n=30648, avg_degree=16.0, seed=3349)),
    ("er", dict(n=5021, avg_degree=8.0, seed=3350)),
    ("er", dict(n=25357, avg_degree=8.0, seed=3351)),
    ("er", dict(n=3815899, avg_degree=16.0, seed=3352)),
    ("er", dict(n=11453, avg_degree=4.0, seed=3353)),
    ("er", dict(n=6248, avg_degree=8.0, seed=3354)),
    ("er", dict(n=956449, avg_degree=16.0, seed=3355)),
    ("er", dict(n=284227, avg_degree=16.0, seed=3356)),
    ("er", dict(n=29545, avg_degree=24.0, seed=3357)),
    ("er", dict(n=201500, avg_degree=8.0, seed=3358)),
    ("er", dict(n=3222166, avg_degree=16.0, seed=3359)),
    ("er", dict(n=193327, avg_degree=4.0, seed=3360)),
    ("er", dict(n=6454, avg_degree=24.0, seed=3361)),
    ("er", dict(n=11002, avg_degree=32.0, seed=3362)),
    ("er", dict(n=818826, avg_degree=24.0, seed=3363)),
    ("er", dict(n=241704, avg_degree=8.0, seed=3364)),
    ("er", dict(n=406580, avg_degree=16.0, seed=3365)),
    ("er", dict(n=862735, avg_degree=32.0, seed=3366)),
    ("er", dict(n=126197, avg_degree=4.0, seed=3367)),
    ("er", dict(n=2465928, avg_degree=8.0, seed=3368)),
    ("growing", dict(n=166675, k=2, seed=3369)),
    ("growing", dict(n=23044, k=8, seed=3370)),
    ("growing", dict(n=22955, k=2, seed=3371)),
    ("growing", dict(n=246975, k=3, seed=3372)),
    ("growing", dict(n=24185, k=4, seed=3373)),
    ("growing", dict(n=528442, k=2, seed=3374)),
    ("growing", dict(n=39949, k=4, seed=3375)),
    ("growing", dict(n=212426, k=9, seed=3376)),
    ("growing", dict(n=3913326, k=5, seed=3377)),
    ("growing", dict(n=20296, k=3, seed=3378)),
    ("growing", dict(n=75703, k=8, seed=3379)),
    ("growing", dict(n=72357, k=5, seed=3380)),
    ("growing", dict(n=357319, k=7, seed=3381)),
    ("growing", dict(n=35261, k=5, seed=3382)),
    ("powerlaw", dict(n=106358, degree=10, exponent=2.68, seed=3383, directed=True)),
    ("powerlaw", dict(n=4417328, degree=5, exponent=2.85, seed=3384)),
    ("powerlaw", dict(n=17499, degree=15, exponent=2.19, seed=3385)),
    ("powerlaw", dict(n=1303197, degree=29, exponent=2.08, seed=3386, directed=True)),
    ("powerlaw", dict(n=128149, degree=27, exponent=2.47, seed=3387)),
    ("powerlaw", dict(n=24630, degree=29, exponent=2.81, seed=3388)),
    ("powerlaw", dict(n=54496, degree=27, exponent=2.36, seed=3389, directed=True)),
    ("powerlaw", dict(n=24551, degree=30, exponent=2.09, seed=3390)),
    ("powerlaw", dict(n=44877, degree=14, exponent=2.59, seed=3391)),
    ("powerlaw", dict(n=294034, degree=19, exponent=2.84, seed=3392, directed=True)),
    ("powerlaw", dict(n=3454994, degree=10, exponent=2.99, seed=3393)),
    ("powerlaw", dict(n=427365, degree=29, exponent=2.9, seed=3394)),
    ("powerlaw", dict(n=242992, degree=21, exponent=2.57, seed=3395, directed=True)),
    ("powerlaw", dict(n=38201, degree=25, exponent=2.21, seed=3396)),
    ("powerlaw", dict(n=3556891, degree=4, exponent=2.62, seed=3397)),
    ("powerlaw", dict(n=1227235, degree=26, exponent=2.69, seed=3398, directed=True)),
    ("smallworld", dict(n=1888466, k=9, beta=0.099, seed=3399)),
    ("smallworld", dict(n=12498, k=8, beta=0.013, seed=3400)),
    ("smallworld", dict(n=95130, k=10, beta=0.189, seed=3401)),
    ("smallworld", dict(n=34205, k=6, beta=0.279, seed=3402)),
    ("smallworld", dict(n=3099492, k=6, beta=0.013, seed=3403)),
    ("smallworld", dict(n=620721, k=7, beta=0.255, seed=3404)),
    ("smallworld", dict(n=8511, k=12, beta=0.084, seed=3405)),
    ("smallworld", dict(n=1379262, k=9, beta=0.459, seed=3406)),
    ("bipartite", dict(left=5227, right=147931, edges=1560008, seed=3407)),
    ("bipartite", dict(left=5108, right=474088, edges=3822392, seed=3408)),
    ("bipartite", dict(left=5416, right=573979, edges=1289056, seed=3409)),
    ("bipartite", dict(left=5215, right=435689, edges=2918576, seed=3410)),
    ("bipartite", dict(left=1558, right=3029, edges=23707, seed=3411)),
    ("bipartite", dict(left=4226, right=1440760, edges=4785403, seed=3412)),
    ("bipartite", dict(left=7554, right=194420, edges=2184049, seed=3413)),
    ("bipartite", dict(left=34906, right=678204, edges=7776723, seed=3414)),
    ("bipartite", dict(left=31665, right=452404, edges=3413355, seed=3415)),
    ("bipartite", dict(left=7248, right=111992, edges=1018704, seed=3416)),
    ("layers", dict(count=31, width=3861, k=12, seed=3417)),
    ("layers", dict(count=55, width=7877, k=16, seed=3418, directed=True)),
    ("layers", dict(count=19, width=8303, k=14, seed=3419, directed=True)),
    ("layers", dict(count=60, width=40906, k=15, seed=3420, directed=True)),
    ("layers", dict(count=38, width=2898, k=10, seed=3421)),
    ("layers", dict(count=58, width=3128, k=12, seed=3422, directed=True)),
    ("layers", dict(count=22, width=5994, k=15, seed=3423, directed=True)),
    ("layers", dict(count=89, width=3899, k=12, seed=3424, directed=True)),
    ("layers", dict(count=96, width=3399, k=9, seed=3425)),
    ("layers", dict(count=8, width=25439, k=13, seed=3426, directed=True)),
    ("stars", dict(n=61144, hubs=3, links=2, seed=3427)),
    ("stars", dict(n=49642, hubs=1, links=3, seed=3428)),
    ("stars", dict(n=105037, hubs=3, links=1, seed=3429)),
    ("stars", dict(n=80316, hubs=6, links=2, seed=3430)),
    ("stars", dict(n=32480, hubs=3, links=1, seed=3431)),
    ("stars", dict(n=912251, hubs=74, links=3, seed=3432)),
    ("tree", dict(n=160283, arity=167, seed=3433)),
    ("tree", dict(n=414500, arity=58, seed=3434)),
    ("tree", dict(n=27358, arity=17, seed=3435)),
    ("tree", dict(n=826828, arity=376, seed=3436)),
    ("tree", dict(n=1834338, arity=31, seed=3437)),
    ("hubs", dict(n=64856, degree=4, hubs=3, share=0.355, seed=3438)),
    ("hubs", dict(n=244024, degree=5, hubs=27, share=0.444, seed=3439)),
    ("hubs", dict(n=56136, degree=3, hubs=22, share=0.083, seed=3440)),
    ("hubs", dict(n=79532, degree=2, hubs=11, share=0.159, seed=3441)),
    ("hubs", dict(n=21861, degree=6, hubs=6, share=0.033, seed=3442)),
    ("cliques", dict(count=40, size=488, seed=3443)),
    ("cliques", dict(count=21, size=295, seed=3444)),
    ("cliques", dict(count=32, size=41, seed=3445)),
    ("cliques", dict(count=142, size=271, seed=3446)),
    ("moves", dict(dims=(90, 90), radius=4, seed=3447)),
    ("moves", dict(dims=(600, 600), radius=2, seed=3448)),
    ("moves", dict(dims=(350, 350), radius=3, seed=3449)),
    ("moves", dict(dims=(60, 60, 60), radius=1, seed=3450)),
    ("moves", dict(dims=(120, 120, 60), radius=1, seed=3451)),
    ("regular", dict(n=887148, k=12, seed=3452)),
    ("regular", dict(n=1055425, k=24, seed=3453)),
    ("regular", dict(n=24404, k=24, seed=3454)),
    ("regular", dict(n=256495, k=36, seed=3455)),
    ("rmatn", dict(n=38032, degree=4, seed=3456, directed=True)),
    ("rmatn", dict(n=985602, degree=4, seed=3457, directed=True)),
    ("rmatn", dict(n=39112, degree=32, seed=3458)),
    ("rmatn", dict(n=120884, degree=16, seed=3459)),
    ("rmatn", dict(n=10789, degree=4, seed=3460)),
    ("rmatn", dict(n=34379, degree=4, seed=3461, directed=True)),
    ("rmatn", dict(n=2548509, degree=8, seed=3462, directed=True)),
    ("rmatn", dict(n=166842, degree=16, seed=3463)),
    ("rmatn", dict(n=175726, degree=4, seed=3464)),
    ("rmatn", dict(n=4804, degree=16, seed=3465)),
    ("rmatn", dict(n=84704, degree=16, seed=3466, directed=True)),
    ("rmatn", dict(n=759337, degree=32, seed=3467, directed=True)),
    ("rmatn", dict(n=459462, degree=32, seed=3468)),
    ("rmatn", dict(n=1216601, degree=32, seed=3469)),
    ("rmatn", dict(n=359036, degree=8, seed=3470)),
    ("rmatn", dict(n=13088, degree=4, seed=3471, directed=True)),
    ("rmatn", dict(n=100742, degree=8, seed=3472, directed=True)),
    ("rmatn", dict(n=6059, degree=24, seed=3473)),
    ("rmatn", dict(n=60841, degree=8, seed=3474)),
    ("rmatn", dict(n=290437, degree=8, seed=3475)),
    ("rmatn", dict(n=72782, degree=4, seed=3476, directed=True)),
    ("rmatn", dict(n=454788, degree=16, seed=3477, directed=True)),
    ("rmatn", dict(n=5351, degree=32, seed=3478)),
    ("rmatn", dict(n=69906, degree=16, seed=3479)),
    ("rmatn", dict(n=10441, degree=32, seed=3480)),
    ("rmatn", dict(n=921827, degree=32, seed=3481, directed=True)),
    ("rmatn", dict(n=143403, degree=8, seed=3482, directed=True)),
    ("rmatn", dict(n=78042, degree=24, seed=3483)),
    ("rmatn", dict(n=24123, degree=4, seed=3484)),
    ("rmatn", dict(n=92991, degree=8, seed=3485)),
    ("rmatn", dict(n=1646772, degree=8, seed=3486, directed=True)),
    ("rmatn", dict(n=1648235, degree=8, seed=3487, directed=True)),
    ("rmatn", dict(n=9695, degree=16, seed=3488)),
    ("rmatn", dict(n=102917, degree=8, seed=3489)),
    ("rmatn", dict(n=42841, degree=16, seed=3490)),
    ("rmatn", dict(n=848827, degree=8, seed=3491, directed=True)),
    ("rmatn", dict(n=250991, degree=32, seed=3492, directed=True)),
    ("rmatn", dict(n=73903, degree=4, seed=3493)),
    ("rmatn", dict(n=14765, degree=8, seed=3494)),
    ("rmatn", dict(n=1967696, degree=8, seed=3495)),
    ("er", dict(n=9177, avg_degree=4.0, seed=3496)),
    ("er", dict(n=555959, avg_degree=16.0, seed=3497)),
    ("er", dict(n=25894, avg_degree=24.0, seed=3498)),
    ("er", dict(n=81917, avg_degree=4.0, seed=3499)),
    ("er", dict(n=140033, avg_degree=16.0, seed=3500)),
    ("er", dict(n=1048864, avg_degree=32.0, seed=3501)),
    ("er", dict(n=1708838, avg_degree=8.0, seed=3502)),
    ("er", dict(n=47076, avg_degree=24.0, seed=3503)),
    ("er", dict(n=116046, avg_degree=4.0, seed=3504)),
    ("er", dict(n=24097, avg_degree=16.0, seed=3505)),
    ("er", dict(n=36039, avg_degree=16.0, seed=3506)),
    ("er", dict(n=184236, avg_degree=16.0, seed=3507)),
    ("er", dict(n=9423, avg_degree=32.0, seed=3508)),
    ("er", dict(n=1184350, avg_degree=8.0, seed=3509)),
    ("er", dict(n=187373, avg_degree=32.0, seed=3510)),
    ("er", dict(n=236202, avg_degree=8.0, seed=3511)),
    ("rmat", dict(scale=19, edge_factor=6, a=0.5, b=0.225, c=0.225, seed=3512)),
    ("rmat", dict(scale=20, edge_factor=10, a=0.6, b=0.175, c=0.175, seed=3513)),
    ("rmat", dict(scale=19, edge_factor=10, a=0.71, b=0.12, c=0.12, seed=3514)),
    ("rmat", dict(scale=17, edge_factor=4, a=0.44, b=0.255, c=0.255, seed=3515)),
    ("rmat", dict(scale=17, edge_factor=6, a=0.63, b=0.16, c=0.16, seed=3516)),
    ("rmat", dict(scale=17, edge_factor=6, a=0.71, b=0.12, c=0.12, seed=3517)),
]


def shape_edges(kind, kw, rng):
    """(vertices, sources, targets) of the generated shapes beside R-MAT, grids and
    Erdos-Renyi: rings with rewired edges, preferential attachment, power-law
    degrees, lattices whose moves reach every cell within a radius, chains of
    cliques, stars (every leaf names `links` hubs in turn), trees, sparse random graphs
    with hubs that name a share of all vertices, separate random components, layers
    whose vertices name k of the next layer, random bipartite and regular graphs."""
    if kind == "rmatn":  # over the next power of two, its first n ids
        n, m = kw["n"], kw["n"] * kw["degree"]
        s, t = np.zeros(m, np.int64), np.zeros(m, np.int64)
        for _ in range((n - 1).bit_length()):
            x = rng.random(m)
            s = 2 * s + (x >= 0.76)
            t = 2 * t + (((x >= 0.57) & (x < 0.76)) | (x >= 0.95))
        ok = (s < n) & (t < n)
        return n, s[ok], t[ok]
    if kind == "smallworld":
        n, k = kw["n"], kw["k"]
        s = np.repeat(np.arange(n), k)
        t = (s + np.tile(np.arange(1, k + 1), n)) % n
        moved = rng.random(n * k) < kw["beta"]
        return n, s, np.where(moved, rng.integers(0, n, n * k), t)
    if kind == "growing":
        n, k = kw["n"], kw["k"]
        s = np.repeat(np.arange(n), k)
        return n, s, (rng.random(n * k) ** 2 * s).astype(np.int64)
    if kind == "powerlaw":
        n, m = kw["n"], kw["n"] * kw["degree"] // (1 if kw.get("directed") else 2)
        c = np.cumsum(np.arange(1, n + 1) ** (-1.0 / (kw["exponent"] - 1.0)))
        return n, np.searchsorted(c, rng.random(m) * c[-1]), np.searchsorted(c, rng.random(m) * c[-1])
    if kind == "moves":
        dims, r = kw["dims"], kw["radius"]
        n = int(np.prod(dims))
        at = np.unravel_index(np.arange(n), dims)
        src, dst = [], []
        for move in np.ndindex(*([2 * r + 1] * len(dims))):
            d = np.array(move) - r
            if tuple(d) <= (0,) * len(dims):
                continue
            to = [x + int(y) for x, y in zip(at, d)]
            ok = np.logical_and.reduce([(x >= 0) & (x < e) for x, e in zip(to, dims)])
            src.append(np.nonzero(ok)[0])
            dst.append(np.ravel_multi_index([x[ok] for x in to], dims))
        return n, np.concatenate(src), np.concatenate(dst)
    if kind == "cliques":
        n, c = kw["count"] * kw["size"], kw["size"]
        i = np.arange(n)
        pairs = [(i[i % c + j < c], i[i % c + j < c] + j) for j in range(1, c)]
        pairs.append((i[:-1][i[:-1] % c == c - 1], i[1:][i[:-1] % c == c - 1]))
        return n, np.concatenate([p[0] for p in pairs]), np.concatenate([p[1] for p in pairs])
    if kind == "stars":
        n, h = kw["n"], kw["hubs"]
        leaves = np.arange(h, n)
        s = np.repeat(leaves, kw.get("links", 1))
        t = (s + np.tile(np.arange(kw.get("links", 1)), n - h)) % h
        return n, s, t
    if kind == "tree":
        child = np.arange(1, kw["n"])
        return kw["n"], child, (child - 1) // kw["arity"]
    if kind == "hubs":
        n, m, h = kw["n"], kw["n"] * kw["degree"] // 2, int(kw["n"] * kw["share"])
        s = np.concatenate([rng.integers(0, n, m), np.repeat(np.arange(kw["hubs"]), h)])
        return n, s, rng.integers(0, n, len(s))
    if kind == "components":
        n, c = kw["count"] * kw["size"], kw["size"]
        s = rng.integers(0, n, n * kw["degree"] // 2)
        return n, s, s // c * c + rng.integers(0, c, len(s))
    if kind == "layers":
        w, k = kw["width"], kw["k"]
        s = np.repeat(np.arange((kw["count"] - 1) * w), k)
        return kw["count"] * w, s, (s // w + 1) * w + rng.integers(0, w, len(s))
    if kind == "bipartite":
        n = kw["left"] + kw["right"]
        return n, rng.integers(0, kw["left"], kw["edges"]), kw["left"] + rng.integers(0, kw["right"], kw["edges"])
    if kind == "regular":
        n, k = kw["n"], kw["k"]
        return n, np.tile(np.arange(n), k // 2), np.concatenate([rng.permutation(n) for _ in range(k // 2)])
    raise ValueError(kind)


def family(name: str) -> str:
    """Generator family of a training graph's name: rmat, rmat-dir, grid, er or another shape's kind."""
    if name.startswith("rmat"):
        return "rmat-dir" if name.endswith("-dir") else "rmat"
    return name.split("-")[0]


def make_graph(kind, kw):
    import graphgen as gg
    if kind == "rmat":
        kw = dict(kw)
        return gg.rmat(kw.pop("scale"), kw.pop("edge_factor"), **kw)
    if kind == "grid":
        return gg.grid(kw["rows"], kw["cols"], kw["drop"], seed=kw["seed"], permute=True)
    if kind == "er":
        return gg.erdos_renyi(kw["n"], kw["avg_degree"], seed=kw["seed"])
    directed = bool(kw.get("directed"))
    if kind == "rmatcut":  # R-MAT over the next power of two, its first n ids
        n = kw["n"]
        g = gg.rmat((n - 1).bit_length(), kw["edge_factor"], seed=kw["seed"], directed=directed)
        s, t = np.repeat(np.arange(g.n), np.diff(g.off)), g.idx
        ok = (s < n) & (t < n)
        return gg.from_edges(n, s[ok], t[ok], symmetrize=not directed,
                             name=f"rmatcut-n{n}-seed{kw['seed']}" + ("-dir" if directed else ""))
    rng = np.random.default_rng(kw["seed"])
    n, s, t = shape_edges(kind, kw, rng)
    p = np.arange(n) if kind == "rmatn" else rng.permutation(n)  # ids in random order
    return gg.from_edges(n, p[s], p[t], symmetrize=not directed,
                         name=f"{kind}-n{n}-seed{kw['seed']}" + ("-dir" if directed else ""))


def collect(out: str, roots_per_graph: int = 4, reps: int = 3, max_levels: int = 16384, graphs=None):
    import graphgen as gg
    import torch
    import paper_1708_01159_gb300 as bfs
    bfs.build()
    torch.cuda.set_device(0)
    graphs = graphs or TRAIN_GRAPHS
    cols = ["graph", "root", "level"] + list(FEATURES) + [f"ms_{v}" for v in VARIANTS] + ["tree_variant"]
    with open(out, "w", newline="") as fh:
        w = csv.writer(fh)
        w.writerow(cols)
        for kind, kw in graphs:
            t0 = time.time()
            g = make_graph(kind, kw)
            name = g.name
            roots = gg.sample_roots(g, roots_per_graph, seed=kw["seed"] + 500, giant=True)
            flags = 0 if kw.get("directed") else bfs.BFS_SYMMETRIC
            with bfs.Graph(g.off, g.idx, flags) as G:
                for r in roots:
                    feats, ms, tv = bfs.bfs_profile_levels(G.handle, int(r), reps=reps, capacity=max_levels)
                    for L in range(feats.shape[0]):
                        w.writerow([name, int(r), L] + [int(x) for x in feats[L]] + [f"{x:.5f}" for x in ms[L]]
                                   + [int(tv[L])])
            fh.flush()
            print(f"{name}: {len(roots)} roots in {time.time() - t0:.1f}s", file=sys.stderr, flush=True)


def load(csv_path: str):
    import gzip
    fh = gzip.open(csv_path, "rt") if csv_path.endswith(".gz") else open(csv_path)
    rows = list(csv.DictReader(fh))
    graph = np.array([r["graph"] for r in rows])
    root = np.array([int(r["root"]) for r in rows])
    level = np.array([int(r["level"]) for r in rows])
    X = np.array([[int(r[f]) for f in FEATURES] for r in rows], dtype=np.int64).reshape(-1, NUM_FEATURES)
    T = np.array([[float(r[f"ms_{v}"]) for v in VARIANTS] for r in rows]).reshape(-1, NUM_VARIANTS)
    return graph, root, level, X, leader_times(X, T)


# On graphs whose out-degrees are at most LEADER_DEGREE the drivers expand a
# level of at most LEADER_EDGES frontier edges on one cluster whichever push
# the tree picks (bfs_small.cuh: 16 blocks x 1088 edges); the timing harness
# times the whole-grid kernels. leader_times takes the cluster's time from the
# 4096^2 grid (1.9 us below 2,000 frontier edges, 3.6 us at 15,900).
LEADER_DEGREE, LEADER_EDGES = 8, 16 * 1088


def leader_times(X, T):
    """The times with every push variant's replaced by the cluster's where it runs."""
    e = X[:, FEATURES.index("frontier_edges")]
    small = (X[:, FEATURES.index("deg_max")] <= LEADER_DEGREE) & (e <= LEADER_EDGES)
    push = [i for i, v in enumerate(VARIANTS) if v != "pull"]
    T = T.copy()
    T[np.ix_(small, push)] = (1.8e-3 + 0.115e-6 * e[small])[:, None]
    return T


def split_by_graph(graph, test_frac=0.3, seed=0):
    names = sorted(set(graph.tolist()))
    rng = np.random.default_rng(seed)
    rng.shuffle(names)
    k = max(1, int(round(test_frac * len(names))))
    test = set(names[:k])
    return np.array([g not in test for g in graph]), sorted(test)


def level_weights(T, trav, weighting):
    """Sample weights. 'uniform': the paper's plain classification. 'regret':
    a level weighs its spread of times (slowest minus fastest), so splits go
    where a wrong choice costs most. 'relregret': that spread divided by the
    traversal's per-level-optimal time, the level's share of the traversal
    slowdown that Table 2 averages. 'cost': as 'relregret', with the spread cut
    at 16 times the level's best (one whole-graph pull of a hub's list costs a
    thousand levels) and the step to the second best added, so that close calls
    count too, and R-MAT and Erdos-Renyi graphs counted twice; its tree is pruned
    and its leaves are labelled by the full costs (fit)."""
    if weighting == "uniform":
        return np.ones(len(T))
    spread = T.max(axis=1) - T.min(axis=1) + 1e-5
    if weighting == "regret":
        return spread
    tot = traversal_optimum(T, trav)
    if weighting == "cost":
        s = np.sort(T, axis=1)
        w = (s[:, 1] - s[:, 0] + np.minimum(s[:, -1] - s[:, 0], 16 * s[:, 0])) / tot + 1e-6
        return w * frequency(trav)
    return spread / tot


def frequency(trav):
    """How often a traversal's graph counts under the 'cost' weighting: R-MAT (whole,
    cut, directed) and Erdos-Renyi, what the library is mostly used on, twice."""
    twice = {t: family(str(t).split("/")[0]) in ("rmat", "rmat-dir", "er") for t in set(trav)}
    return np.array([2.0 if twice[t] else 1.0 for t in trav])


def traversal_optimum(T, trav):
    """For every level, the per-level-optimal time of its whole traversal."""
    tot = {}
    for k, t in zip(trav, T.min(axis=1)):
        tot[k] = tot.get(k, 0.0) + t
    return np.array([tot[k] for k in trav])


# The library decides a tree's tests on graph features for each graph, and evaluates
# what is left in its bit-parallel form, held in shared memory, when that has at
# most 64 leaves (more are walked node by node in global memory, about 1 us per
# level). Up to 33 a warp tests all of its nodes at once: of 96 leaves in all the
# graphs of the training set keep 26 in the middle and 31 at most. (192 leaves, of
# which 36 were kept, cost 1 to 2.5 % of small traversals over 64 and 20.)
MAX_LEAVES = 96
GROWN_LEAVES = 1000  # of a tree that is pruned


def fit(X, T, feature_idx, max_depth=8, min_samples_leaf=8, weighting="regret", trav=None, max_leaves=MAX_LEAVES):
    """CART with Gini impurity (Section 2.1); labels: the fastest variant per level.
    Under the 'cost' weighting the tree is grown larger and pruned back by cost
    (prune), and each leaf is labelled with the variant of least total cost over its
    levels (each level's times over its traversal's optimum) instead of the heaviest
    class: clf.leaf_label_, by node."""
    from sklearn.tree import DecisionTreeClassifier
    y = T.argmin(axis=1)
    w = level_weights(T, trav if trav is not None else np.zeros(len(T)), weighting)
    grown = max(GROWN_LEAVES, max_leaves) if weighting == "cost" else max_leaves
    clf = DecisionTreeClassifier(criterion="gini", max_depth=max_depth, min_samples_leaf=min_samples_leaf,
                                 max_leaf_nodes=grown, random_state=0)
    clf.fit(X[:, feature_idx], y, sample_weight=w)
    if weighting == "cost":
        cost = np.zeros((clf.tree_.node_count, T.shape[1]))
        np.add.at(cost, clf.apply(X[:, feature_idx].astype(np.float32)),
                  T * (frequency(trav) / traversal_optimum(T, trav))[:, None])
        prune(clf, cost, max_leaves)
    return clf


def prune(clf, cost, max_leaves):
    """Cost-complexity pruning (Breiman et al. 1984) with the levels' cost in place of
    the misclassification rate: while there are too many leaves, the subtree whose
    leaves save the least cost each over its root as a leaf is cut. cost: by leaf and
    variant. Sets clf.leaf_label_ (the variant of least cost of every leaf left)."""
    left, right = clf.tree_.children_left, clf.tree_.children_right
    order, todo = [], [0]
    while todo:
        i = todo.pop()
        order.append(i)
        if left[i] >= 0:
            todo += [left[i], right[i]]
    parent = np.full(len(left), -1)
    leaves = np.ones(len(left), dtype=np.int64)
    for i in reversed(order):
        if left[i] >= 0:
            cost[i] = cost[left[i]] + cost[right[i]]
            parent[left[i]] = parent[right[i]] = i
    own = cost.min(axis=1)
    sub = own.copy()
    for i in reversed(order):
        if left[i] >= 0:
            sub[i] = sub[left[i]] + sub[right[i]]
            leaves[i] = leaves[left[i]] + leaves[right[i]]
    inner = {i for i in order if left[i] >= 0}
    while leaves[0] > max_leaves:
        cut = min(inner, key=lambda i: ((own[i] - sub[i]) / (leaves[i] - 1), i))
        up, gain, gone = parent[cut], own[cut] - sub[cut], leaves[cut] - 1
        todo = [cut]
        while todo:
            i = todo.pop()
            if i in inner:
                inner.discard(i)
                todo += [left[i], right[i]]
        sub[cut], leaves[cut] = own[cut], 1
        while up >= 0:
            sub[up] += gain
            leaves[up] -= gone
            up = parent[up]
    kept = [i for i in order if i == 0 or parent[i] in inner]
    clf.leaf_label_ = {int(i): int(cost[i].argmin()) for i in kept if i not in inner}


def export(clf, feature_idx, path, meta=""):
    """Integer tree text: 'feature threshold left right value' per node."""
    t = clf.tree_
    labels = getattr(clf, "leaf_label_", None)
    nodes, todo = [], [0]  # what is left of a pruned tree
    while todo:
        i = todo.pop()
        nodes.append(i)
        if t.children_left[i] >= 0 and not (labels and i in labels):
            todo += [t.children_left[i], t.children_right[i]]
    nodes.sort()  # a parent before its children
    number = {i: k for k, i in enumerate(nodes)}
    lines = []
    for i in nodes:
        if t.children_left[i] < 0 or (labels and i in labels):
            v = t.value[i][0]
            order = np.argsort(v)[::-1]
            cls = clf.classes_
            top = int(cls[order[0]])
            tie = len(order) > 1 and math.isclose(float(v[order[0]]), float(v[order[1]]), rel_tol=1e-9)
            lines.append(f"-1 0 -1 -1 {labels[i] if labels else -1 if tie else top}")
        else:
            f = int(feature_idx[t.feature[i]])
            lines.append(f"{f} {int(math.floor(t.threshold[i]))} {number[t.children_left[i]]} "
                         f"{number[t.children_right[i]]} -1")
    with open(path, "w") as fh:
        fh.write("# Decision tree trained on per-level GB300 timings (CART, Gini).\n")
        for m in meta.splitlines():
            fh.write(f"# {m}\n")
        fh.write("# Features: " + ", ".join(f"{i} {f}" for i, f in enumerate(FEATURES)) + "\n")
        fh.write("# Classes: " + ", ".join(f"{i} {v}" for i, v in enumerate(VARIANTS)) + "\n")
        fh.write(f"bfs-tree 1 {len(nodes)}\n")
        fh.write("\n".join(lines) + "\n")


def read_tree(path):
    from paper_1708_01159_gb300.buildlib import parse_tree_text
    rows = parse_tree_text(open(path).read())
    return [{"f": f, "t": t, "l": l, "r": r, "v": v} for f, t, l, r, v in rows]


def walk(nodes, x):
    i = 0
    while nodes[i]["f"] >= 0:
        i = nodes[i]["l"] if x[nodes[i]["f"]] <= nodes[i]["t"] else nodes[i]["r"]
    return nodes[i]["v"]


def schedule_time(nodes, X, T, level):
    """Per-level choice with the unknown rule; returns the chosen variants."""
    out = np.empty(len(X), dtype=np.int64)
    for i in range(len(X)):
        v = walk(nodes, X[i])
        if v < 0:
            v = out[i - 1] if level[i] > 0 else LEVEL0_DEFAULT
        out[i] = v
    return out


def evaluate(graph, root, level, X, T, nodes, mask=None):
    """Table-2-shaped summary over traversals: slowdown vs the per-level optimum."""
    if mask is None:
        mask = np.ones(len(X), bool)
    keys = sorted(set(zip(graph[mask].tolist(), root[mask].tolist())))
    pred = schedule_time(nodes, X, T, level)
    rows = {"predicted": [], "best_fixed": []}
    for v in VARIANTS:
        rows[v] = []
    fixed_by_graph = {}
    for gname in set(graph[mask].tolist()):
        sel = mask & (graph == gname)
        fixed_by_graph[gname] = int(T[sel].sum(axis=0).argmin())
    acc_hits = 0
    for gname, r in keys:
        sel = np.nonzero(mask & (graph == gname) & (root == r))[0]
        opt = T[sel].min(axis=1).sum()
        rows["predicted"].append(T[sel, pred[sel]].sum() / opt)
        rows["best_fixed"].append(T[sel, fixed_by_graph[gname]].sum() / opt)
        for k, v in enumerate(VARIANTS):
            rows[v].append(T[sel, k].sum() / opt)
        acc_hits += int((pred[sel] == T[sel].argmin(axis=1)).sum())
    summary = {}
    for k, vals in rows.items():
        a = np.array(vals)
        summary[k] = {"optimal": float((a < 1.0 + 1e-9).mean()), "1-2x": float(((a >= 1) & (a <= 2)).mean()),
                      ">5x": float((a > 5).mean()), ">20x": float((a > 20).mean()), "average": float(a.mean()),
                      "worst": float(a.max())}
    summary["level_accuracy"] = acc_hits / int(mask.sum())
    summary["traversals"] = len(keys)
    return summary


def cross_validate(graph, root, level, X, T, folds=6, depths=(6, 8, 10), feature_sets=None,
                   weightings=("uniform", "regret", "relregret", "cost")):
    """Mean held-out slowdown vs the per-level optimum, k folds split by graph."""
    import tempfile
    names = sorted(set(graph.tolist()))
    rng = np.random.default_rng(1)
    rng.shuffle(names)
    fold_of = {nm: i % folds for i, nm in enumerate(names)}
    fold = np.array([fold_of[g] for g in graph])
    trav = np.array([f"{g}/{r}" for g, r in zip(graph, root)])
    for fs in sorted(feature_sets or FEATURE_SETS):
        for wt in weightings:
            for depth in depths:
                slow, worst, best_fixed = [], 0.0, []
                for k in range(folds):
                    tr, te = fold != k, fold == k
                    fidx = np.array(FEATURE_SETS[fs])
                    clf = fit(X[tr], T[tr], fidx, depth, 8, wt, trav[tr])
                    with tempfile.NamedTemporaryFile("w", suffix=".tree", delete=False) as fh:
                        path = fh.name
                    export(clf, fidx, path)
                    s = evaluate(graph, root, level, X, T, read_tree(path), te)
                    os.unlink(path)
                    slow.append(s["predicted"]["average"] * s["traversals"])
                    best_fixed.append(s["best_fixed"]["average"] * s["traversals"])
                    worst = max(worst, s["predicted"]["worst"])
                n = len(set(trav.tolist()))
                print(f"features={fs:5s} weighting={wt:9s} depth={depth:2d}: held-out mean {sum(slow) / n:.3f}x "
                      f"worst {worst:.2f}x (best fixed {sum(best_fixed) / n:.3f}x)", flush=True)


def level_split(graph, root, level, X, T, test_frac=0.3, seed=0, depths=(6, 8, 10)):
    """The paper's protocol (Section 2.1, Section 4.4): a random 70/30 split over
    levels, pooled across graphs, scored by held-out per-level accuracy (the
    predicted variant is the fastest one). Levels of one traversal are
    correlated, so this flatters a tree compared with the split by graph; it is
    reported for comparability. Also the share of held-out levels whose
    prediction is within 10 % of the fastest time."""
    rng = np.random.default_rng(seed)
    te = np.zeros(len(X), bool)
    te[rng.permutation(len(X))[: int(round(test_frac * len(X)))]] = True
    tr = ~te
    trav = np.array([f"{g}/{r}" for g, r in zip(graph, root)])
    y = T.argmin(axis=1)
    rows = np.nonzero(te)[0]
    for fs in sorted(FEATURE_SETS):
        fidx = np.array(FEATURE_SETS[fs])
        for wt in ("uniform", "relregret"):
            for depth in depths:
                clf = fit(X[tr], T[tr], fidx, depth, 8, wt, trav[tr])
                pred = clf.predict(X[te][:, fidx])
                acc = float((pred == y[te]).mean())
                near = float((T[rows, pred] <= 1.1 * T[rows].min(axis=1)).mean())
                print(f"features={fs:5s} weighting={wt:9s} depth={depth:2d}: held-out level accuracy {acc:.3f}, "
                      f"within 10 % of the fastest {near:.3f} ({int(te.sum())} of {len(X)} levels)", flush=True)


def holdout_families(graph, root, level, X, T, features="ext_io", weighting="relregret", depth=8, min_leaf=8):
    """Section 4.4's generality question on generated families: for each
    family (R-MAT, directed R-MAT, grid, Erdos-Renyi) in turn, train on the
    other families only and evaluate on this one; per family, the tree's and
    the best fixed variant's traversal time relative to the per-level optimum."""
    import tempfile
    fam = np.array([family(g) for g in graph])
    trav = np.array([f"{g}/{r}" for g, r in zip(graph, root)])
    fidx = np.array(FEATURE_SETS[features])
    print(f"held-out family (features={features} weighting={weighting} depth={depth}):")
    print(f"{'family':10s} {'traversals':>10s} {'tree/opt':>9s} {'worst':>7s} {'best fixed/opt':>15s} "
          f"{'tree <= best fixed':>19s}")
    out = {}
    for f in sorted(set(fam.tolist())):
        tr, te = fam != f, fam == f
        clf = fit(X[tr], T[tr], fidx, depth, min_leaf, weighting, trav[tr])
        with tempfile.NamedTemporaryFile("w", suffix=".tree", delete=False) as fh:
            path = fh.name
        export(clf, fidx, path)
        nodes = read_tree(path)
        os.unlink(path)
        pred = schedule_time(nodes, X, T, level)
        keys = sorted(set(zip(graph[te].tolist(), root[te].tolist())))
        fixed = {g: int(T[te & (graph == g)].sum(axis=0).argmin()) for g in set(graph[te].tolist())}
        rt, rb, wins = [], [], 0
        for g, r in keys:
            sel = np.nonzero(te & (graph == g) & (root == r))[0]
            opt = T[sel].min(axis=1).sum()
            t_tree = T[sel, pred[sel]].sum()
            t_fix = T[sel, fixed[g]].sum()
            rt.append(t_tree / opt)
            rb.append(t_fix / opt)
            wins += int(t_tree <= t_fix * 1.0001)
        out[f] = {"traversals": len(keys), "tree_over_opt": float(np.mean(rt)), "worst": float(np.max(rt)),
                  "best_fixed_over_opt": float(np.mean(rb)), "tree_le_best_fixed": wins / len(keys)}
        print(f"{f:10s} {len(keys):10d} {np.mean(rt):8.3f}x {np.max(rt):6.2f}x {np.mean(rb):14.3f}x "
              f"{wins / len(keys):18.0%}", flush=True)
    return out


def print_table(summary, file=sys.stdout):
    print(f"traversals: {summary['traversals']}, per-level accuracy: {summary['level_accuracy']:.3f}", file=file)
    print(f"{'algorithm':14s} {'optimal':>8s} {'1-2x':>7s} {'>5x':>6s} {'>20x':>6s} {'average':>8s} {'worst':>8s}",
          file=file)
    for k in ["predicted", "best_fixed"] + list(VARIANTS):
        s = summary[k]
        print(f"{k:14s} {s['optimal']:8.2%} {s['1-2x']:7.2%} {s['>5x']:6.2%} {s['>20x']:6.2%} "
              f"{s['average']:7.2f}x {s['worst']:7.2f}x", file=file)


def main():
    p = argparse.ArgumentParser()
    sub = p.add_subparsers(dest="cmd", required=True)
    c = sub.add_parser("collect")
    c.add_argument("--out", required=True)
    c.add_argument("--roots", type=int, default=4)
    c.add_argument("--reps", type=int, default=3)
    t = sub.add_parser("train")
    t.add_argument("--csv", required=True)
    t.add_argument("--out", required=True)
    t.add_argument("--features", default="ext", choices=sorted(FEATURE_SETS))
    t.add_argument("--max-depth", type=int, default=8)
    t.add_argument("--min-leaf", type=int, default=8)
    t.add_argument("--weighting", default="relregret", choices=["regret", "uniform", "relregret", "cost"])
    t.add_argument("--all-graphs", action="store_true", help="train on every graph (no held-out split)")
    v = sub.add_parser("cv", help="k-fold cross-validation by graph over feature sets and weightings")
    v.add_argument("--csv", required=True)
    v.add_argument("--folds", type=int, default=6)
    v.add_argument("--features", nargs="*", default=None, choices=sorted(FEATURE_SETS))
    v.add_argument("--weightings", nargs="*", default=["uniform", "regret", "relregret", "cost"])
    ls = sub.add_parser("level-split", help="the paper's random 70/30 split over levels: held-out accuracy")
    ls.add_argument("--csv", required=True)
    h = sub.add_parser("holdout", help="leave each graph family out in turn (Section 4.4 generality)")
    h.add_argument("--csv", required=True)
    h.add_argument("--features", default="ext_io", choices=sorted(FEATURE_SETS))
    h.add_argument("--weighting", default="relregret", choices=["regret", "uniform", "relregret", "cost"])
    h.add_argument("--max-depth", type=int, default=8)
    e = sub.add_parser("evaluate")
    e.add_argument("--csv", required=True)
    e.add_argument("--tree", required=True)
    a = p.parse_args()
    if a.cmd == "collect":
        collect(a.out, a.roots, a.reps)
        return
    graph, root, level, X, T = load(a.csv)
    if a.cmd == "train":
        fidx = np.array(FEATURE_SETS[a.features])
        train_mask, test_graphs = split_by_graph(graph)
        if a.all_graphs:
            train_mask = np.ones(len(graph), bool)
        trav = np.array([f"{g}/{r}" for g, r in zip(graph, root)])
        clf = fit(X[train_mask], T[train_mask], fidx, a.max_depth, a.min_leaf, a.weighting, trav[train_mask])
        meta = (f"features={a.features} max_depth={a.max_depth} min_samples_leaf={a.min_leaf} "
                f"weighting={a.weighting}\nlevels={int(train_mask.sum())} "
                f"held-out graphs={'none' if a.all_graphs else ','.join(test_graphs)}")
        export(clf, fidx, a.out, meta)
        nodes = read_tree(a.out)
        print("train:")
        print_table(evaluate(graph, root, level, X, T, nodes, train_mask))
        if not a.all_graphs:
            print("held-out graphs:", ", ".join(test_graphs))
            print_table(evaluate(graph, root, level, X, T, nodes, ~train_mask))
    elif a.cmd == "cv":
        cross_validate(graph, root, level, X, T, a.folds, feature_sets=a.features, weightings=a.weightings)
    elif a.cmd == "level-split":
        level_split(graph, root, level, X, T)
    elif a.cmd == "holdout":
        holdout_families(graph, root, level, X, T, a.features, a.weighting, a.max_depth)
    else:
        print_table(evaluate(graph, root, level, X, T, read_tree(a.tree)))


if __name__ == "__main__":
    main()

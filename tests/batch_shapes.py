"""Batches, by the vertices + entries of their graphs, that reach every shape of
the batch kernel on a GPU of 152 SMs: clusters of 16, 8, 4 and 2 blocks for
some of the graphs and single blocks for the rest, 512 and 1024 threads (with 8
colour classes)."""
SHAPES = {
    # name: (sizes, blocks of a cluster, threads, graphs run by clusters)
    "c16_512": ([120000, 60000, 40000, 3000], 16, 512, 2),
    "c16_1024": ([1900000], 16, 1024, 1),
    "c8_512": ([60000] * 5 + [30000] * 5 + [22000] * 10 + [2000] * 10, 8, 512, 10),
    "c8_1024": ([120000] * 30, 8, 1024, 17),
    "c4_512": ([30000] * 8 + [14500] * 8 + [10500] * 8 + [3000] * 40, 4, 512, 16),
    "c2_512": ([14000] * 10 + [7500] * 10 + [5000] * 70, 2, 512, 20),
    "c1_512": ([10000] * 120, 1, 512, 0),
    "c1_1024": ([110000] * 4 + [2000] * 116, 1, 1024, 0),
}

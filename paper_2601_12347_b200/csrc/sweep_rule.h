// When a hop's messages are swept instead of pushed: plain C++, used on the host (is the sweep in the chain?) and on the
// device (which of the two delivers?).
//
// Microseconds, fitted to whole hops: a push pays per float delivered (0.65 ps where the accumulator stays in L2, 0.79
// where it does not) and per sender, whose list a warp takes up after the one before (0.8 ns); a sweep per edge of the graph
// (5.5 ps) and per row added up (4 ps and 0.29 per float), and is taken where it saves a tenth: hops at the line lose the
// launch.  Measured, kernels of a hop, push / sweep: 1.0 M messages of 256 floats from 34 K senders on a graph of 1.2 M edges
// 230 / 164 us, 1.1 M of 40 floats from 80 K senders 135 / 110; 124 M edges: 24 M of 48 floats 968 / 1102 and of 256 5690 / 1990,
// 33 M of 128 floats 2134 / 1261; 115 M edges: 39 M of 128 floats 4095 / 1728.  (Fitted before the sweep had its registers and
// its L1: 49 M of 44 floats from 9 K senders, 115 M edges, 1451 / 1269, are still left to the push.)
#pragma once

#ifdef __CUDACC__
#define RP_RULE __host__ __device__ inline
#else
#define RP_RULE inline
#endif

namespace rp {

constexpr long long WALK_TWICE = 160ll << 20;   // bytes of rows from which a walk is made twice (see TicketWalk)

// The device's choice, by what the hop does carry.
RP_RULE bool sweep_pays(double msgs, double senders, double edges, double vertices, int width) {
    const bool outgrows = vertices * width * 4.0 > (double)WALK_TWICE;
    const double push = 5.0 + 1e-6 * msgs * width * (outgrows ? 0.79 : 0.65) + 0.8e-3 * senders;
    const double sweep = 30.0 + 1e-6 * (5.5 * edges + msgs * (4.0 + 0.29 * width));
    return sweep < 0.9 * push;
}

// The host's: both forms come into the chain if twice what the hop carried in the batch before would be swept (unknown: if all
// edges from all vertices would), and stay in it while four times as much would: a stream of batches that differ by less than
// a factor two keeps one chain, also near the line (each change of the chain costs a batch launched kernel by kernel and a
// capture, a quarter to half a millisecond).
inline bool sweep_may_pay(bool known, bool armed, double msgs, double senders, double edges, double vertices, int width) {
    const double by = armed ? 4.0 : 2.0;
    return known ? sweep_pays(by * msgs, by * senders, edges, vertices, width) : sweep_pays(edges, vertices, edges, vertices, width);
}

// What ctl->pull says of a hop.
enum { PUSHED = 0, SWEPT = 1, SWEEP_MARKED = 2 };

// Of a hop that is swept because the caller wants it (RIPPLE_SCATTER_PULL): every in-list of the graph, or only the lists of
// its frontier, which a walk over the senders' out-lists marks first.  124 M edges, walk and sweep of the frontier / sweep of
// everything: 9 messages of 100 floats 116 / 440 us, 22 K of 256 floats 250 / 480, 2.3 M 830 / 815, 19 M 1810 / 1630, 122 M of
// 48 floats 4890 / 4170; 115 M edges: 0.4 M of 256 floats 1109 / 1070.
RP_RULE bool sweep_reads_all(double msgs, double edges) { return 8.0 * msgs >= edges; }

}  // namespace rp

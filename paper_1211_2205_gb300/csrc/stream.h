// Interface of the FP64 streamed half-step pass (2D P_N).
#pragma once
#include <cstdint>
#include <vector>

#include "host_math.h"
#include "internal.h"

namespace starmap {

// One stage of a pass for one output kind (R or I): the inputs whose
// differences it adds and the target it completes (kernels_stream.cu).
struct StreamRec {
    double p0, np;          // weights of the previous input of the order: the target completed, the next-order target
    double pm, n0;          // weights of the stage's input: the target completed, the next-order target
    int16_t own, other;     // input component of the kind and of the other kind, in its grid (-1: none)
    int16_t out;            // component completed, in its grid (-1: none)
    int16_t src;            // its source slot (-1: none)
    int8_t cls;             // its decay class
    int8_t pre, post, store;    // partial-sum slots: read before the stage, read at its end for the next
                            // stage's target, written at its end (-1: none)
    int8_t op;              // the kind of stage (StreamOp)
    int8_t pad[3];
};
static_assert(sizeof(StreamRec) == 48, "staged in 16-byte pieces");
// Kinds of stages: with both inputs, with that of the kind or of the other
// kind alone (m' = 0), without inputs; HEAD: the first of an order, TOP: of
// the highest input order (no next-order targets).
enum StreamOp {
    OP_NONE, OP_FULL, OP_FULL_TOP, OP_HEAD, OP_HEAD_TOP, OP_OWN, OP_OWN_TOP, OP_OWN_HEAD, OP_OTHER, OP_OTHER_TOP,
    OP_OTHER_HEAD, OP_TAIL, OP_TAIL_TOP
};

// One output of a pass by its own: its input pairs, up to four, in the order
// in which the stages add them: (l - 1, q - 1), (l - 1, q), (l + 1, q),
// (l + 1, q + 1); bit k of t: pair k enters by t (the first and third of
// those), else by s.
struct PairRec {
    double w[4];
    int16_t own[4], other[4];   // input components (-1: none)
    int16_t out, src;
    int8_t cls, count, t;
    int8_t pad[9];
};
static_assert(sizeof(PairRec) == 64, "four 16-byte loads");

struct StreamTables;

struct StreamArgs {
    GridDev<double> g[4];
    long pitch;
    int p[2];
    int P, which;           // pass parity, coefficient set
    double* const* src;     // source arrays [ny][cp] by slot
};

// Tables of both passes, on the host; null where the order's couplings do not
// have the structure the kernel streams.  Returns 0 or -4.
int stream_build(const SystemMatrices& sys, const std::vector<char>& frozen, double dx, double dy, StreamTables** out);
// Decay classes and source slots of the components; uploads the tables, into
// one buffer that the first call allocates.  Returns 0 or -4.
int stream_update(StreamTables* t, const std::vector<int>& comp_class, const std::vector<int>& src_slot);
void stream_destroy(StreamTables* t);
int stream_pass(const StreamTables* t, const StreamArgs& a, void* stream);

}  // namespace starmap

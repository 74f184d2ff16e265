// solve_ordered_a.cu -- the ordered solver of Taylor-Green steps, N + 1 in {4, 7, 10}.
#include "solver_ordered.cuh"

int sem_solve_ordered_a(const SolveParams<8> &p, int n, int sms, cudaStream_t s)
{
    switch (n) {
        case 4: return ordered::launch<4>(p, sms, s);
        case 7: return ordered::launch<7>(p, sms, s);
        case 10: return ordered::launch<10>(p, sms, s);
        default: return SEM_ERR_ARG;
    }
}

int sem_solve_ordered_tables_a(int n, const double *D) { return solver_upload_tables(n, D); }
